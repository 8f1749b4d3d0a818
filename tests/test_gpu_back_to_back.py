"""Compression and the first generated tokens enqueued back to back: kernels of a call may start while the ones ahead of them
on the stream still run, and the first decode step must nevertheless see the finished caches.  The same calls with a
synchronisation after each give the same outputs and caches, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2406_13035_b200 import binding as B

pytestmark = pytest.mark.gpu

STEPS = 3


def _prompt(rng, L, hq, hkv, P, d, td, dev):
    g = torch.Generator(device=dev).manual_seed(rng)
    Q = torch.randn(L, 1, hq, P, d, generator=g, device=dev).to(td)
    # keys in few clusters: most evicted tokens merge
    c = torch.randn(L, 1, hkv, 8, d, generator=g, device=dev)
    K = c[:, :, :, torch.randint(0, 8, (P,), generator=g, device=dev)] + 0.1 * torch.randn(L, 1, hkv, P, d, generator=g, device=dev)
    V = torch.randn(L, 1, hkv, P, d, generator=g, device=dev).to(td)
    q = torch.randn(STEPS, L, 1, hq, d, generator=g, device=dev).to(td)
    k, v = (torch.randn(STEPS, L, 1, hkv, d, generator=g, device=dev).to(td) for _ in range(2))
    return Q, K.to(td), V, q, k, v


def _run(synced, mode, prompts, L, hq, hkv, P, d, dtype, rho):
    ctx = B.D2OContext(B.make_config(n_layers=L, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                     max_new_tokens=8, rho=rho, n_sink=1, window=8, min_budget=16, density_temp=1e30))
    done = []
    for Q, K, V, q, k, v in prompts:
        out = torch.empty_like(q)
        ctx.d2o_layer_stats_layers(0, L, list(Q), list(K))
        ctx.d2o_layer_budgets()
        torch.cuda.synchronize()
        ctx.d2o_prefill_compress_layers(0, L, list(K), list(V))
        if synced:
            torch.cuda.synchronize()
        if mode == "steps":
            ctx.d2o_decode_steps(0, L, STEPS, q, k, v, out)
        else:
            for s in range(STEPS):
                for l in range(L):
                    ctx.d2o_decode_step(l, l + 1, q[s, l], k[s, l], v[s, l], out[s, l])
                    if synced:
                        torch.cuda.synchronize()
        torch.cuda.synchronize()
        tabs = ctx.tables()
        done.append((out, [ctx.slice_state(l, 0, h, tabs) for l in range(L) for h in range(hkv)]))
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()
    return done


@pytest.mark.parametrize("mode", ["steps", "by layer"])
@pytest.mark.parametrize("L,hq,hkv,P,d,dtype,rho", [
    (1, 8, 8, 300, 64, "f32", 0.3),
    (1, 32, 8, 1500, 128, "bf16", 0.2),
    (4, 32, 8, 700, 128, "bf16", 0.3),
    (16, 8, 8, 400, 128, "f16", 0.25),
    (4, 8, 8, 200, 64, "f32", 1.0),        # nothing is evicted: the gather is the last kernel of the compression
    (16, 16, 8, 150, 128, "bf16", 1.0)])
def test_first_steps_behind_a_compression(cuda_device, mode, L, hq, hkv, P, d, dtype, rho):
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    # the second prompt finds the first conversation's lengths and step counters
    prompts = [_prompt(s, L, hq, hkv, P, d, td, cuda_device) for s in (1, 2)]
    want = _run(True, mode, prompts, L, hq, hkv, P, d, dtype, rho)
    for _ in range(5):
        got = _run(False, mode, prompts, L, hq, hkv, P, d, dtype, rho)
        for (wo, ws), (go, gs) in zip(want, got):
            assert torch.equal(wo.view(torch.uint8), go.view(torch.uint8))
            for a, b in zip(ws, gs):
                assert a["len"] == b["len"] and np.float32(a["tau"]).tobytes() == np.float32(b["tau"]).tobytes()
                for key in ("pos", "score", "rnorm", "K", "V"):
                    assert torch.equal(a[key].view(torch.uint8), b[key].view(torch.uint8)), key


@pytest.mark.parametrize("L,B_,hkv,P", [(4, 1, 8, 512), (32, 16, 32, 1024)])
def test_budgets_are_complete_on_return(cuda_device, L, B_, hkv, P):
    """d2o_layer_budgets synchronises its stream: what it uploads for the calls behind it is there for calls on any stream.
    The larger case uploads half a megabyte of work lists."""
    d, td = 64, torch.float16
    ctx = B.D2OContext(B.make_config(n_layers=L, batch=B_, n_q_heads=hkv, n_kv_heads=hkv, d_head=d, dtype="f16", prompt_len=P,
                                     max_new_tokens=2, rho=0.3, n_sink=1, min_budget=16))
    Q = torch.randn(B_, hkv, P, d, device=cuda_device).to(td)
    ctx.d2o_layer_stats_layers(0, L, [Q] * L, [Q] * L)
    call, handle, stream = ctx.lib.d2o_layer_budgets, ctx.handle, torch.cuda.current_stream()
    at, done = stream.cuda_stream, []
    for _ in range(50):
        status = call(handle, None, at)
        done.append(status == 0 and stream.query())
    assert all(done)
    assert ctx.d2o_get_stats().error_word == 0
    ctx.close()
