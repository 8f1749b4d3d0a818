"""Inverse norms of the prompt rows in the similarity of 16-bit keys (Eq. 9): summed per 16-byte segment and then as a tree,
as the norms of the retained rows are.

The keys make the norm readable from the maximum similarity.  Retained are the unit rows e_0 .. e_{d-1}, whose norm is
exactly 1; every evicted row has one element of 16 and all others below it, so its largest similarity is 16 / |k|, a scaling
by a power of two that rounds nowhere.  Products of 16-bit values are exact in fp32, and so is numpy's restatement of the
sums, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2406_13035_b200 import binding as B

pytestmark = pytest.mark.gpu


def _inverse_norms(x):
    """x: float32 [n, d].  Segments of eight in element order, then pairs d/16, d/32, .. segments apart."""
    sq = (x * x).reshape(x.shape[0], -1, 8)
    s = np.zeros(sq.shape[:2], np.float32)
    for i in range(8):
        s = s + sq[:, :, i]
    while s.shape[1] > 1:
        h = s.shape[1] // 2
        s = s[:, :h] + s[:, h:]
    return np.float32(1) / np.sqrt(s[:, 0])


@pytest.mark.parametrize("dtype,d,P", [("bf16", 128, 700), ("bf16", 64, 391), ("f16", 128, 513), ("f16", 64, 1025)])
def test_prompt_norms_are_summed_as_a_tree(cuda_device, dtype, d, P):
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    ctx = B.D2OContext(B.make_config(n_layers=1, batch=1, n_q_heads=1, n_kv_heads=1, d_head=d, dtype=dtype, prompt_len=P,
                                     max_new_tokens=2, rho=d / P, n_sink=0, window=1, min_budget=8, density_temp=1e30,
                                     max_budget=P))
    rng = np.random.default_rng(P)
    K = torch.tensor(rng.uniform(-15, 15, (P, d)), dtype=torch.float32).to(td)
    K[torch.arange(P), torch.tensor(rng.integers(0, d, P))] = 16.0
    K[P - d:] = torch.eye(d, dtype=torch.float32).to(td)          # the last d rows: one window row, the others by score
    K = K.to(cuda_device)[None, None].contiguous()
    ctx.d2o_layer_stats(0, K, K)
    ctx.colsum(0).copy_((torch.arange(P, device=cuda_device) >= P - d).float()[None, None])
    ctx.density().fill_(1.0)
    assert int(ctx.d2o_layer_budgets()[0, 0, 0]) == d
    ctx.d2o_prefill_compress(0, K, K)
    idx, mx, _ = ctx.evict_lists(0, 0, P - d)
    np.testing.assert_array_equal(idx.numpy(), np.arange(P - d))
    want = np.float32(16) * _inverse_norms(K[0, 0, :P - d].float().cpu().numpy())
    np.testing.assert_array_equal(mx.numpy().view(np.uint32), want.view(np.uint32))
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()
