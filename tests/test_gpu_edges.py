"""Kernels that divide their work by size, at the sizes where the division changes: the decode kernel with one cluster of
CTAs per slice (against the float64 oracle, with the tolerances of parity.py), the selection of the retained positions across
its blocks of 4096 and with ties (exact), and the uncompressed decode around its row groups."""
import dataclasses
import math

import numpy as np
import pytest
import torch

from paper_2406_13035_b200 import binding as B
from paper_2406_13035_b200 import workloads as W

from parity import assert_report, close, np64, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,rho,hq,hkv,d,dtype", [
    (40, 0.5, 1, 1, 64, "f32"),            # fewer rows than warps in the cluster
    (129, 0.99, 2, 2, 128, "f16"),         # 127 - 129 rows on two CTAs, in copies of 32
    (642, 0.5, 4, 1, 128, "bf16"),         # 321 rows: four CTAs instead of two
    (640, 0.5, 40, 40, 64, "f16"),         # more slices than a quarter of the SMs: two
    (1501, 0.7, 8, 1, 128, "bf16"),        # eight heads per slice
    (1900, 0.9, 2, 1, 128, "f32"),         # rows that need eight CTAs
    (2600, 0.97, 1, 1, 128, "f16")])       # more rows than four CTAs hold
def test_decode_cluster(P, rho, hq, hkv, d, dtype):
    wl = dataclasses.replace(W.CONFIGS["cfg0"], n_layers=1, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype,
                             prompt_len=P, rho=rho, decode_steps=4, min_budget=8)
    rep = run_parity(wl, slices=[(0, 0, h) for h in sorted({0, hkv - 1})])
    assert rep.steps == 4
    assert_report(rep, dtype)


@pytest.mark.parametrize("P,rho,hq,hkv,d,dtype", [
    (40, 0.5, 1, 1, 64, "f32"), (129, 0.99, 2, 2, 128, "f16"), (642, 0.5, 4, 1, 128, "bf16"), (640, 0.5, 40, 40, 64, "f16"),
    (1501, 0.7, 8, 1, 128, "bf16"), (1900, 0.9, 2, 1, 128, "f32"), (2600, 0.97, 1, 1, 128, "f16"),
    (800, 0.99, 32, 32, 128, "bf16"), (333, 0.6, 64, 64, 64, "bf16"), (700, 0.8, 16, 8, 64, "f16"), (517, 0.9, 16, 4, 64, "f32"),
    (450, 0.7, 16, 2, 128, "f16"), (40, 0.5, 4, 1, 128, "bf16"), (129, 0.99, 4, 2, 128, "f16"), (640, 0.5, 80, 40, 64, "f16"),
    (640, 0.99, 72, 36, 128, "bf16")])
def test_decode_cluster_values(cuda_device, P, rho, hq, hkv, d, dtype):
    """Attention spread over all rows (logits of variance 1), so that every value row counts: outputs of one step against
    float64 on the rows the cache holds.  An output is the rounding of something within e of the reference.  A logit errs by a
    few 2^-24 of the magnitudes it sums (about 7), a weight by as much; over the rows the errors are of random sign, so that
    the output errs by about 2e-7 of its root mean square: e = 1.5e-6 of it.  With several heads on bf16 caches the weights
    enter as two bf16 terms, up to 2^-17 off: 4e-6, e = 3e-5.  A missing row would be 1e-3 or more."""
    ctx = B.D2OContext(B.make_config(n_layers=1, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                     max_new_tokens=4, rho=rho, n_sink=1, min_budget=8, density_temp=1e30))
    td, G = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]], hq // hkv
    g = torch.Generator(device=cuda_device).manual_seed(P)
    draw = lambda *s: torch.randn(*s, generator=g, device=cuda_device).to(td)
    K, V = draw(1, hkv, P, d), draw(1, hkv, P, d)
    ctx.d2o_layer_stats(0, draw(1, hq, P, d), K)
    ctx.d2o_layer_budgets()
    ctx.d2o_prefill_compress(0, K, V)
    for _ in range(2):
        q, k, v = draw(1, 1, hq, d), draw(1, 1, hkv, d), draw(1, 1, hkv, d)
        tabs = ctx.tables()
        refs = []
        for h in range(hkv):
            st = ctx.slice_state(0, 0, h, tabs)
            Kh, Vh = np.r_[np64(st["K"]), np64(k[0, :, h])], np.r_[np64(st["V"]), np64(v[0, :, h])]
            x = np64(q[0, 0, h * G:(h + 1) * G]) @ Kh.T / math.sqrt(d)
            w = np.exp(x - x.max(1, keepdims=True))
            refs.append(w @ Vh / w.sum(1, keepdims=True))
        ref = np.concatenate(refs)
        out = torch.empty_like(q)
        ctx.d2o_decode_step(0, 1, q, k, v, out)
        got, rms = np64(out[0, 0]), math.sqrt(np.mean(ref * ref))
        e = (3e-5 if dtype == "bf16" and G > 1 else 1.5e-6) * rms
        lo, hi = np64(torch.tensor(ref - e).to(td)), np64(torch.tensor(ref + e).to(td))
        assert np.all((lo <= got) & (got <= hi)), (float(np.max(np.abs(got - ref) / rms)), int(np.sum((got < lo) | (got > hi))))
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()


@pytest.mark.parametrize("P,hq,d,dtype", [(65, 4, 128, "bf16"), (65, 2, 64, "f32"), (225, 1, 128, "bf16"), (225, 8, 64, "bf16")])
def test_decode_cluster_warp_without_a_finite_logit(cuda_device, P, hq, d, dtype):
    """The new token's tile of 16 rows holds no other row, and its logits overflow to -inf for every head: the token has
    weight 0 in its own step and in the next, and the outputs are those of the other rows (bounds as above)."""
    ctx = B.D2OContext(B.make_config(n_layers=1, batch=1, n_q_heads=hq, n_kv_heads=1, d_head=d, dtype=dtype, prompt_len=P,
                                     max_new_tokens=8, rho=(P + 8) / P, n_sink=1, min_budget=8, max_budget=P + 8))
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    g = torch.Generator(device=cuda_device).manual_seed(P)
    draw = lambda *s: torch.randn(*s, generator=g, device=cuda_device).to(td)
    K, V = draw(1, 1, P, d), draw(1, 1, P, d)
    K[..., 0] = 0.0
    ctx.d2o_layer_stats(0, draw(1, hq, P, d), K)
    ctx.d2o_layer_budgets()
    ctx.d2o_prefill_compress(0, K, V)
    Kh, Vh = np64(K[0, 0]), np64(V[0, 0])
    for step in range(2):
        q, k, v = draw(1, 1, hq, d), draw(1, 1, 1, d), draw(1, 1, 1, d)
        q[..., 0] = 64.0
        k[..., 0] = -3e38 if step == 0 else 0.0
        if step > 0:
            Kh, Vh = np.r_[Kh, np64(k[0, 0])], np.r_[Vh, np64(v[0, 0])]
        x = np64(q[0, 0]) @ Kh.T / math.sqrt(d)
        w = np.exp(x - x.max(1, keepdims=True))
        ref = w @ Vh / w.sum(1, keepdims=True)
        out = torch.empty_like(q)
        ctx.d2o_decode_step(0, 1, q, k, v, out)
        e = (3e-5 if dtype == "bf16" and hq > 1 else 1.5e-6) * math.sqrt(np.mean(ref * ref))
        got, lo, hi = np64(out[0, 0]), np64(torch.tensor(ref - e).to(td)), np64(torch.tensor(ref + e).to(td))
        assert np.all((lo <= got) & (got <= hi))
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()


@pytest.mark.parametrize("P", [17, 1023, 4095, 4096, 4097, 8193])
def test_retained_positions_with_ties(cuda_device, P):
    """Scores of seven distinct values over 17 layers (one more than share a launch): retained are the sinks, the window and
    the highest scores, equal ones by the earlier position; every other position is evicted."""
    L, S, sinks, window, d = 17, max(8, P // 5), 1, 4, 64
    ctx = B.D2OContext(B.make_config(n_layers=L, batch=1, n_q_heads=2, n_kv_heads=1, d_head=d, dtype="f16", prompt_len=P,
                                     max_new_tokens=2, rho=S / P, n_sink=sinks, window=window, min_budget=8,
                                     density_temp=1e30, max_budget=P))
    g = torch.Generator(device=cuda_device).manual_seed(P)
    x = torch.randn(L, 1, 2, P, d, generator=g, device=cuda_device).half()
    for l in range(L):
        ctx.d2o_layer_stats(l, x[l], x[l, :, :1])
        ctx.colsum(l).copy_(torch.randint(0, 7, (1, 2, P), generator=g, device=cuda_device).float())
    ctx.density().fill_(1.0)
    ctx.d2o_layer_budgets()
    keys = [x[l, :, :1].contiguous() for l in range(L)]
    ctx.d2o_prefill_compress_layers(0, L, keys, keys)
    tabs = ctx.tables()
    for l in (0, 15, 16):
        score = ctx.colsum(l)[0].sum(0).cpu().numpy()
        st = ctx.slice_state(l, 0, 0, tabs)
        middle = np.arange(sinks, P - st["M"])
        best = middle[np.lexsort((middle, -score[middle]))][:st["S"] - sinks - st["M"]]
        np.testing.assert_array_equal(st["pos"].numpy(), np.sort(np.r_[np.arange(sinks), best, np.arange(P - st["M"], P)]))
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()


@pytest.mark.parametrize("length", [1, 31, 32, 63, 64, 255, 1024])
@pytest.mark.parametrize("dtype,d,G,n", [("f16", 128, 1, 1), ("bf16", 64, 4, 150), ("f32", 128, 2, 3)])
def test_full_decode_lengths(cuda_device, dtype, d, G, n, length):
    """Slices in one wave of CTAs, several CTAs per slice for few of them; fp32 softmax and sums against float64: 2^-24 of
    the logits (below 60) and of the sums, plus the rounding of the stored output, as in parity.py."""
    td = W.TORCH_DTYPES[dtype]
    g = torch.Generator(device=cuda_device).manual_seed(length)
    kc, vc = (torch.randn(n, length + 3, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    q = torch.randn(n, G, d, generator=g, device=cuda_device).to(td)
    k, v = (torch.randn(n, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    out = torch.empty_like(q)
    B.d2o_full_decode_step(kc, vc, length, q, k, v, out)
    K, V = torch.cat([kc[:, :length], k[:, None]], 1).double(), torch.cat([vc[:, :length], v[:, None]], 1).double()
    ref = torch.softmax(q.double() @ K.transpose(1, 2) / math.sqrt(d), -1) @ V
    assert close(np64(out), ref.cpu().numpy(), dtype) <= 1.0


@pytest.mark.parametrize("dtype,d,G,length", [("f16", 128, 1, 200), ("bf16", 64, 4, 65), ("f32", 128, 2, 1000), ("bf16", 128, 8, 1)])
def test_full_decode_non_finite_keys(cuda_device, dtype, d, G, length):
    """A NaN in a cached key reaches every output of its slice, as it does in the softmax; a logit of -inf is weight 0."""
    td, n, row = W.TORCH_DTYPES[dtype], 4, length // 2
    g = torch.Generator(device=cuda_device).manual_seed(length)
    kc, vc = (torch.randn(n, length + 2, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    q = torch.randn(n, G, d, generator=g, device=cuda_device).to(td)
    k, v = (torch.randn(n, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    kc[..., 0], k[:, 0] = 0.0, 0.0
    q[..., 0] = 4.0
    kc[1, row, 1] = float("nan")
    kc[2, row, 0] = -float("inf")
    k[3, 5] = float("nan")
    out = torch.empty_like(q)
    K, V = torch.cat([kc[:, :length], k[:, None]], 1).double(), torch.cat([vc[:, :length], v[:, None]], 1).double()
    B.d2o_full_decode_step(kc, vc, length, q, k, v, out)
    ref = torch.softmax(q.double() @ K.transpose(1, 2) / math.sqrt(d), -1) @ V
    assert torch.isnan(out[1]).all() and torch.isnan(out[3]).all()
    for s in (0, 2):
        assert close(np64(out[s]), ref[s].cpu().numpy(), dtype) <= 1.0
