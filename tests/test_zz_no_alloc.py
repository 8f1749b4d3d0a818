"""The allocation-free entry point against the regular one.

Some users of the library cannot call cudaMalloc while it runs: an inference server whose memory
pool has taken the whole device, or a host application that passes tensors in but keeps its
allocator to itself.  d2o_layer_stats_static serves them with a scratch array that lives inside
the library image.  It runs the kernels of d2o_layer_stats, or for fp32 inputs, whose dot products it cannot
keep, other ones that add in the same order, so the two agree bit for bit (checked
for fp32 inputs, at more lengths in test_gpu_colsum_lengths.py, and for a prompt length that is no multiple of 4) and within the parity tolerance,
also on a second call that finds the first call's leftovers in the scratch array.
The results are checked against the CPU oracle as well, and the free device memory must not move
across the call.
This file sorts last on purpose, so that a run which stops at the first failure has already
been through every other test.
"""
import dataclasses

import pytest
import torch

from paper_2406_13035_b200 import binding as B
from paper_2406_13035_b200 import workloads as W

from parity import make_ctx

pytestmark = pytest.mark.gpu


def _regular(wl, Q, K):
    ctx = make_ctx(wl)
    ctx.d2o_layer_stats(0, Q, K)
    cs = ctx.colsum(0).clone()
    F = ctx.density()[:, 0, :].clone()
    torch.cuda.synchronize()
    ctx.close()
    return cs, F


@pytest.mark.parametrize("name,P,same_kernels", [("cfg0", 300, True), ("cfg2", 777, True), ("cfg2", 512, False)])
def test_static_scratch_entry_matches_regular_entry(cuda_device, name, P, same_kernels):
    import numpy as np
    from oracle import d2o_oracle as O
    from paper_2406_13035_b200 import build
    build.build_library()
    B.load_library()
    base = dataclasses.replace(W.CONFIGS[name], n_layers=1, batch=2, prompt_len=P, decode_steps=1, window=8,
                               max_budget=0)
    for call in range(2):                               # the second call reuses the scratch of the first
        wl = dataclasses.replace(base, seed=base.seed + call)
        Q, K, _ = W.LayerStream(wl, 0, "cuda:0").prompt()
        ref_cs, ref_F = _regular(wl, Q, K)
        cs = torch.full((wl.batch, wl.n_q_heads, P), float("nan"), dtype=torch.float32, device=cuda_device)
        F = torch.full((wl.batch, wl.n_q_heads), float("nan"), dtype=torch.float64, device=cuda_device)
        torch.cuda.synchronize()
        free_before, _ = torch.cuda.mem_get_info()
        B.d2o_layer_stats_static(Q, K, cs, F)
        torch.cuda.synchronize()
        free_after, _ = torch.cuda.mem_get_info()
        assert free_after == free_before                 # nothing was allocated or freed on the device
        torch.testing.assert_close(cs, ref_cs, rtol=2e-4, atol=0)
        torch.testing.assert_close(F, ref_F, rtol=2e-4, atol=0)
        if same_kernels:                                 # same kernels, or (fp32) the same order of the sums: bit-identical
            assert torch.equal(cs, ref_cs) and torch.equal(F, ref_F)
        # against the oracle, on two heads of the second sequence
        Qc, Kc = Q.cpu().double().numpy(), K.cpu().double().numpy()
        for hq in (0, wl.n_q_heads - 1):
            s_ref = O.colsum_scores(Qc[1, hq], Kc[1, hq // wl.group])
            got = cs[1, hq].cpu().double().numpy()
            assert np.max(np.abs(got - s_ref) / np.maximum(np.abs(s_ref), 1e-6)) < 2e-4
            assert abs(float(F[1, hq]) - O.attention_density(s_ref)) <= 2e-4 * O.attention_density(s_ref)


def test_scratch_without_room_for_dot_products(cuda_device):
    """fp32: a scratch that lacks only the room for the dot products (every head's whole tiles, for two layers) is accepted, one that
    lacks a byte more is not; column sums and caches are those of the full scratch, bit for bit."""
    import ctypes as C
    from paper_2406_13035_b200 import build
    build.build_library()
    wl = dataclasses.replace(W.CONFIGS["cfg0"], n_layers=3, batch=1, prompt_len=300, decode_steps=2, window=8, max_budget=0)
    products = 2 * wl.n_q_heads * 15 * 64 * 64 * 4        # 5 tiles of 64 rows: 15 on and below the diagonal
    streams = [W.LayerStream(wl, l, "cuda:0") for l in range(3)]
    Q, K, V = zip(*[s.prompt() for s in streams])

    def results(ctx):
        ctx.d2o_layer_stats_layers(0, 3, Q, K)
        ctx.d2o_layer_budgets()
        ctx.d2o_prefill_compress_layers(0, 3, K, V)
        tabs = ctx.tables()
        return [ctx.colsum(l).clone() for l in range(3)] + [ctx.slice_state(l, 0, h, tabs)["K"] for l in range(3) for h in range(wl.n_kv_heads)]

    full = make_ctx(wl)
    want = results(full)
    lib, cfg = B.load_library(), full.cfg
    sb, xb = B.d2o_workspace_size(cfg)
    small = make_ctx(wl)
    lib.d2o_destroy(small.handle)
    small.scratch[small._scratch_off + xb - products:].fill_(0x5a)
    sp, xp = (t.data_ptr() + off for t, off in ((small.state, small._state_off), (small.scratch, small._scratch_off)))
    h = C.c_void_p()
    st = torch.cuda.current_stream().cuda_stream
    assert lib.d2o_create(C.byref(cfg), sp, sb, xp, xb - products - 256, st, C.byref(h)) == 3
    assert lib.d2o_create(C.byref(cfg), sp, sb, xp, xb - products, st, C.byref(h)) == 0
    small.handle = h
    for a, b in zip(want, results(small)):
        assert torch.equal(a, b)
    torch.cuda.synchronize()
    assert bool((small.scratch[small._scratch_off + xb - products:] == 0x5a).all())      # and left alone
    full.close()
    small.close()


def test_static_scratch_entry_rejects_oversize(cuda_device):
    B.load_library()
    P = B.STATIC_LSE_FLOATS // 8 + 1                    # 1 x 8 heads x P floats: one row too many
    Q = torch.zeros(1, 8, P, 64, dtype=torch.float16, device=cuda_device)
    K = torch.zeros(1, 8, P, 64, dtype=torch.float16, device=cuda_device)
    cs = torch.zeros(1, 8, P, dtype=torch.float32, device=cuda_device)
    F = torch.zeros(1, 8, dtype=torch.float64, device=cuda_device)
    with pytest.raises(B.D2OError) as e:
        B.d2o_layer_stats_static(Q, K, cs, F)
    assert e.value.status == 7
    # more (sequence, head) pairs than a grid has rows
    Q = torch.zeros(1, 65536, 4, 64, dtype=torch.float16, device=cuda_device)
    K = torch.zeros(1, 65536, 4, 64, dtype=torch.float16, device=cuda_device)
    cs = torch.zeros(1, 65536, 4, dtype=torch.float32, device=cuda_device)
    F = torch.zeros(1, 65536, dtype=torch.float64, device=cuda_device)
    with pytest.raises(B.D2OError) as e:
        B.d2o_layer_stats_static(Q, K, cs, F)
    assert e.value.status == 7
