"""Column sums of the prompt attention (Eq. 4) at prompt lengths around the tile edges of the tensor-core kernels and at
lengths that are no multiple of anything, against the attention in float64.

Tolerance: the logits are exact products of 16-bit values summed in fp32 (relative error about d * 2^-24 of the sum of
their magnitudes, here below 4e-6 of a logit of magnitude ~10), one exponential (2^-22) and fp32 / fp64 sums: 2e-5 of a
column sum covers it four times."""
import math

import pytest
import torch

from paper_2406_13035_b200 import binding as B

pytestmark = pytest.mark.gpu


def _reference(Q, K):
    q, k = Q.double(), K.double().repeat_interleave(Q.shape[1] // K.shape[1], 1)
    x = q @ k.transpose(-1, -2) / math.sqrt(Q.shape[-1])
    P = Q.shape[2]
    x = x.masked_fill(torch.ones(P, P, dtype=torch.bool, device=x.device).triu(1), float("-inf"))
    return x, torch.softmax(x, -1).sum(-2)


def _context(dtype, b, hq, hkv, d, P):
    return B.D2OContext(B.make_config(n_layers=1, batch=b, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                      max_new_tokens=8, rho=1.0, n_sink=0, min_budget=1))


@pytest.mark.parametrize("P", [1, 2, 31, 63, 64, 65, 127, 129, 191, 255, 257, 321, 383, 514, 769, 1023, 1281])
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f16", 64)])
def test_colsum_at_any_prompt_length(cuda_device, dtype, d, P):
    b, hq, hkv = 2, 4, 2
    g = torch.Generator(device=cuda_device).manual_seed(P)
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    Q = (1.5 * torch.randn(b, hq, P, d, generator=g, device=cuda_device)).to(td)
    K = torch.randn(b, hkv, P, d, generator=g, device=cuda_device).to(td)
    logits, ref = _reference(Q, K)
    ctx = _context(dtype, b, hq, hkv, d, P)
    ctx.d2o_layer_stats(0, Q, K)
    own = ctx.colsum(0).clone()
    assert float(((own.double() - ref).abs() / ref).max()) < 2e-5
    # the normalisers of the caller's own attention kernel; rounded to fp32 (2^-24 of about 10) by the caller
    ctx.d2o_layer_stats(0, Q, K, torch.logsumexp(logits, -1).float().contiguous())
    assert float(((ctx.colsum(0).double() - ref).abs() / ref).max()) < 2e-5
    assert ctx.d2o_get_stats().error_word == 0
    # the allocation-free entry point runs the same kernels
    cs = torch.empty(b, hq, P, device=cuda_device)
    F = torch.empty(b, hq, dtype=torch.float64, device=cuda_device)
    B.d2o_layer_stats_static(Q, K, cs, F)
    assert torch.equal(cs, own)


@pytest.mark.parametrize("hq,hkv", [(1, 1), (8, 4), (96, 96)])
@pytest.mark.parametrize("P", [1, 63, 64, 65, 128, 129, 300, 513, 960, 1025])
@pytest.mark.parametrize("d", [64, 128])
def test_fp32_colsum_at_any_prompt_length(cuda_device, d, P, hq, hkv):
    """Lengths around one tile, odd and even numbers of strips, and head counts that take one to eight CTAs per pair of
    strips.  An fp32 dot product of magnitudes summing to about 11 errs by a few times 11 * 2^-24: the bound above holds."""
    b = 2
    g = torch.Generator(device=cuda_device).manual_seed(P + hq)
    Q = 1.5 * torch.randn(b, hq, P, d, generator=g, device=cuda_device)
    K = torch.randn(b, hkv, P, d, generator=g, device=cuda_device)
    lens = [P, max(1, (2 * P) // 3)]
    ctx = _context("f32", b, hq, hkv, d, P)
    ctx.d2o_set_prompt_lens(torch.tensor(lens, dtype=torch.int32))
    given = torch.zeros(b, hq, P, device=cuda_device)
    refs = []
    for i, p in enumerate(lens):
        logits, ref = _reference(Q[i:i + 1, :, :p], K[i:i + 1, :, :p])
        given[i, :, :p] = torch.logsumexp(logits[0], -1).float()
        refs.append(ref[0])
    for lse in (None, given):
        ctx.d2o_layer_stats(0, Q, K, lse)
        for i, p in enumerate(lens):
            assert float(((ctx.colsum(0)[i, :, :p].double() - refs[i]).abs() / refs[i]).max()) < 2e-5
    assert ctx.d2o_get_stats().error_word == 0


@pytest.mark.parametrize("b,hq,hkv,d,P,L", [
    (2, 1, 1, 64, 1, 1), (2, 8, 4, 128, 65, 1), (1, 8, 8, 64, 450, 3), (2, 96, 96, 64, 1025, 2), (1, 32, 8, 128, 1999, 2),
    (1, 8, 2, 64, 6001, 2), (1, 16, 16, 64, 5000, 3), (1, 32, 32, 64, 5000, 1), (1, 32, 4, 64, 5300, 2), (1, 12, 12, 64, 9000, 1), (1, 4, 4, 64, 11000, 1),
    (1, 2, 1, 64, 12001, 1)])
def test_fp32_colsum_bits_whoever_computes_them(cuda_device, b, hq, hkv, d, P, L):
    """Products stored (all heads, or in groups, with the room of one layer or of all) or computed twice: the bits are those of the
    allocation-free entry point, which computes them twice."""
    g = torch.Generator(device=cuda_device).manual_seed(P)
    Q = [1.5 * torch.randn(b, hq, P, d, generator=g, device=cuda_device) for _ in range(L)]
    K = [torch.randn(b, hkv, P, d, generator=g, device=cuda_device) for _ in range(L)]
    want, F = torch.empty(L, b, hq, P, device=cuda_device), torch.empty(L, b, hq, dtype=torch.float64, device=cuda_device)
    for l in range(L):
        B.d2o_layer_stats_static(Q[l], K[l], want[l], F[l])
    ctx = B.D2OContext(B.make_config(n_layers=L, batch=b, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype="f32", prompt_len=P,
                                     max_new_tokens=8, rho=1.0 if P < 64 else 0.1, n_sink=0, min_budget=1))
    for one_call in (True, False):
        for l in range(L):
            ctx.colsum(l).zero_()
        if one_call:
            ctx.d2o_layer_stats_layers(0, L, Q, K)
        else:
            for l in range(L):
                ctx.d2o_layer_stats(l, Q[l], K[l])
        assert all(torch.equal(ctx.colsum(l), want[l]) for l in range(L))
        assert torch.equal(ctx.density(), F.permute(1, 0, 2))
    ctx.close()


@pytest.mark.parametrize("h,d,P", [(32, 64, 896), (22, 128, 896), (12, 64, 1500), (64, 64, 500), (2, 64, 1999), (5, 128, 7)])
def test_fp32_given_normalisers_with_every_cluster_size(cuda_device, h, d, P):
    """The column sweep by itself, with one, two, four and eight CTAs to a pair of strips."""
    g = torch.Generator(device=cuda_device).manual_seed(P)
    Q = 1.5 * torch.randn(1, h, P, d, generator=g, device=cuda_device)
    K = torch.randn(1, h, P, d, generator=g, device=cuda_device)
    logits, ref = _reference(Q, K)
    ctx = _context("f32", 1, h, h, d, P)
    ctx.d2o_layer_stats(0, Q, K, torch.logsumexp(logits, -1).float().contiguous())
    assert float(((ctx.colsum(0).double() - ref).abs() / ref).max()) < 2e-5
    ctx.close()


@pytest.mark.parametrize("d,P,key", [(64, 100, 97), (64, 65, 3), (128, 449, 448), (64, 128, 70)])
def test_fp32_keys_with_infinite_elements(cuda_device, d, P, key):
    """A key whose logits are all -inf: its column is 0, every other one is as without it, and nothing comes from the rows past the
    end of the last tile, whose products with it are not numbers."""
    h = 4
    g = torch.Generator(device=cuda_device).manual_seed(P)
    Q = torch.randn(1, h, P, d, generator=g, device=cuda_device)
    K = torch.randn(1, h, P, d, generator=g, device=cuda_device)
    Q[..., 5] = Q[..., 5].abs() + 0.1
    K[:, :, key, 5] = -float("inf")
    logits, ref = _reference(Q, K)
    ref[:, :, key] = 0.0
    ctx = _context("f32", 1, h, h, d, P)
    for _ in range(2):
        ctx.d2o_layer_stats(0, Q, K)
        cs = ctx.colsum(0)
        assert bool((cs[:, :, key] == 0).all())
        others = torch.arange(P, device=cuda_device) != key
        assert float(((cs.double() - ref).abs() / ref)[:, :, others].max()) < 2e-5
    static, F = torch.empty(1, h, P, device=cuda_device), torch.empty(1, h, dtype=torch.float64, device=cuda_device)
    B.d2o_layer_stats_static(Q, K, static, F)
    assert torch.equal(static, cs)
    ctx.close()


def test_work_counter_is_zero_after_every_call(cuda_device):
    """The tensor-core kernels take their work from a counter.  Whatever it holds before a call (as after two calls that
    overlapped), the call after that one computes everything."""
    b, hq, hkv, d, P = 1, 32, 8, 64, 1281                          # 192 items: more than the GPU has SMs
    g = torch.Generator(device=cuda_device).manual_seed(P)
    Q = torch.randn(b, hq, P, d, generator=g, device=cuda_device).bfloat16()
    K = torch.randn(b, hkv, P, d, generator=g, device=cuda_device).bfloat16()
    ctx = _context("bf16", b, hq, hkv, d, P)
    ctx.d2o_layer_stats(0, Q, K)
    want = ctx.colsum(0).clone()
    at = ctx._view(0).density - ctx.state.data_ptr() - 256         # the counter's 256 bytes lie ahead of the densities
    counter = ctx.state[at:at + 8].view(torch.int32)
    assert counter.tolist() == [0, 0]
    for dirty in ([3, 1000], [1 << 20, 1], [7, 0]):
        counter.copy_(torch.tensor(dirty, dtype=torch.int32))
        ctx.d2o_layer_stats(0, Q, K)
        ctx.colsum(0).zero_()
        ctx.d2o_layer_stats(0, Q, K)
        assert torch.equal(ctx.colsum(0), want) and counter.tolist() == [0, 0]
    ctx.close()


@pytest.mark.parametrize("dtype,d,P", [("bf16", 128, 700), ("f16", 64, 513)])
def test_normalisers_far_too_low(cuda_device, dtype, d, P):
    """A row whose normaliser is -inf, or 200 below the true one, contributes +inf to every column it attends to (its
    probabilities are 2^288 and more times too large) and nothing else: no NaN, no finite value, in no place of the tiles."""
    g = torch.Generator(device=cuda_device).manual_seed(P)
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    Q = torch.randn(1, 4, P, d, generator=g, device=cuda_device).to(td)
    K = torch.randn(1, 2, P, d, generator=g, device=cuda_device).to(td)
    logits, _ = _reference(Q, K)
    lse = torch.logsumexp(logits, -1)
    at = (P * 3) // 4                                              # from here on the columns see no such row
    low = lse.clone()
    low[0, 0, at - 1] = -float("inf")
    low[0, 1, at - 1] -= 200.0
    low[0, 2, 17] = -float("inf")
    ref = torch.exp(logits - lse[..., None]).sum(-2)
    ctx = _context(dtype, 1, 4, 2, d, P)
    ctx.d2o_layer_stats(0, Q, K, low.float().contiguous())
    cs = ctx.colsum(0)[0]
    for h, n in ((0, at), (1, at), (2, 18), (3, 0)):
        assert torch.isposinf(cs[h, :n]).all()
        assert float(((cs[h, n:].double() - ref[0, h, n:]).abs() / ref[0, h, n:]).max()) < 2e-5
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()
