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


@pytest.mark.parametrize("hq,hkv,P,d,dtype,rho", [
    (32, 8, 700, 128, "bf16", 0.3), (32, 8, 2000, 128, "bf16", 0.4), (16, 16, 300, 128, "f16", 0.5), (8, 8, 400, 64, "f32", 0.4)])
def test_outputs_of_a_layer_are_the_queries_of_the_next(cuda_device, hq, hkv, P, d, dtype, rho):
    """The inputs of a step are still being written when its kernel starts: they are read behind the wait."""
    L, td = 12, B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    Q, K, V, q, k, v = _prompt(5, L, hq, hkv, P, d, td, cuda_device)

    def run(synced):
        ctx = B.D2OContext(B.make_config(n_layers=L, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                         max_new_tokens=8, rho=rho, n_sink=1, window=8, min_budget=16, density_temp=1e30))
        ctx.d2o_layer_stats_layers(0, L, list(Q), list(K))
        ctx.d2o_layer_budgets()
        ctx.d2o_prefill_compress_layers(0, L, list(K), list(V))
        out = torch.zeros(STEPS, L, 1, hq, d, dtype=td, device=cuda_device)
        for s in range(STEPS):
            for l in range(L):
                ctx.d2o_decode_step(l, l + 1, q[s, 0] if l == 0 else out[s, l - 1], k[s, l], v[s, l], out[s, l])
                if synced:
                    torch.cuda.synchronize()
        assert ctx.d2o_get_stats().error_word == 0
        ctx.close()
        return out

    want = run(True)
    for _ in range(5):
        assert torch.equal(want.view(torch.uint8), run(False).view(torch.uint8))


@pytest.mark.parametrize("hq,hkv,P,d,dtype", [(32, 8, 500, 128, "bf16"), (8, 8, 300, 64, "f32")])
def test_step_counters_in_any_order_of_calls(cuda_device, hq, hkv, P, d, dtype):
    """Who writes a slice's step counter depends on the call behind it: other layers, the same ones, a chain of steps, another
    stream, a new prompt."""
    L, td = 4, B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    one = lambda *layers: [(l, l + 1) for l in layers]
    tokens = [one(0, 1, 2, 3), one(0, 1, 2, 3), one(3, 1, 0, 2), [(0, 4)], [(0, 4)], one(1, 0, 3, 2), [(0, 2), (2, 4)], [(0, 2), (2, 4)],
              "chain", one(2, 3, 0, 1), "side stream", one(0, 1, 2, 3), "chain", "new prompt", one(0, 1, 2, 3), one(1, 2, 3, 0)]
    prompts = [_prompt(seed, L, hq, hkv, P, d, td, cuda_device) for seed in (7, 8)]
    g = torch.Generator(device=cuda_device).manual_seed(9)
    q = torch.randn(40, L, 1, hq, d, generator=g, device=cuda_device).to(td)
    k, v = (torch.randn(40, L, 1, hkv, d, generator=g, device=cuda_device).to(td) for _ in range(2))

    def run(synced):
        ctx = B.D2OContext(B.make_config(n_layers=L, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                         max_new_tokens=40, rho=0.3, n_sink=1, window=8, min_budget=16, density_temp=1e30))
        out = torch.zeros_like(q)
        side = torch.cuda.Stream()
        torch.cuda.synchronize()

        def wait():
            if synced:
                torch.cuda.synchronize()

        def prompt(Q, K, V, *_):
            ctx.d2o_layer_stats_layers(0, L, list(Q), list(K))
            ctx.d2o_layer_budgets()
            ctx.d2o_prefill_compress_layers(0, L, list(K), list(V))
            wait()

        def calls(t, ranges):
            for l0, l1 in ranges:
                ctx.d2o_decode_step(l0, l1, q[t, l0:l1], k[t, l0:l1], v[t, l0:l1], out[t, l0:l1])
                wait()

        prompt(*prompts[0])
        t = 0
        for token in tokens:
            if token == "new prompt":
                prompt(*prompts[1])
                continue
            if token == "chain":
                ctx.d2o_decode_steps(0, L, 3, q[t:t + 3], k[t:t + 3], v[t:t + 3], out[t:t + 3])
                wait()
                t += 3
                continue
            if token == "side stream":
                # layers in turn on two streams, each behind the call before
                for i, r in enumerate(one(0, 1, 2, 3, 0, 1, 2, 3)):
                    here, there = torch.cuda.current_stream(), side
                    if i % 3 == 1:
                        there.wait_stream(here)
                        with torch.cuda.stream(there):
                            calls(t + i // L, [r])
                        here.wait_stream(there)
                    else:
                        calls(t + i // L, [r])
                t += 2
                continue
            calls(t, token)
            t += 1
        torch.cuda.synchronize()
        assert ctx.d2o_get_stats().error_word == 0
        tabs = ctx.tables()
        state = [ctx.slice_state(l, 0, h, tabs) for l in range(L) for h in range(hkv)]
        ctx.close()
        return out, state

    want, ws = run(True)
    for _ in range(3):
        got, gs = run(False)
        assert torch.equal(want.view(torch.uint8), got.view(torch.uint8))
        for a, b in zip(ws, gs):
            assert all(torch.equal(a[key].view(torch.uint8), b[key].view(torch.uint8)) for key in ("pos", "score", "rnorm", "K", "V"))


@pytest.mark.parametrize("hq,hkv,d,dtype,pair", [(32, 8, 128, "bf16", False), (16, 16, 128, "f16", False), (16, 16, 64, "f32", False),
                                                  (32, 8, 128, "bf16", True)])
def test_step_counters_of_stacks_on_both_decode_kernels(cuda_device, hq, hkv, d, dtype, pair):
    """Layers with small caches step on clusters and leave their step counters to the next call; layers with large ones step on one
    CTA per slice.  The counters are written whichever kernel comes next, and the results are those of synchronised calls."""
    L, B_, P, tokens = 6, 4, 2400, 5
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    g = torch.Generator(device=cuda_device).manual_seed(P)
    Q, K, V = (torch.randn(L, B_, h, P, d, generator=g, device=cuda_device).to(td) for h in (hq, hkv, hkv))
    q = torch.randn(tokens, L, B_, hq, d, generator=g, device=cuda_device).to(td)
    k, v = (torch.randn(tokens, L, B_, hkv, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    row = 2 * d * (4 if dtype == "f32" else 2) * B_ * hkv                  # bytes of one row of every slice of a layer
    small, large = 12e6 / row, 26e6 / row                                  # on either side of the 20 MB where the kernels change
    big = (1, 2, 4)
    calls = [(0, 1), (1, 3), (3, 4), (4, 5), (5, 6)] if pair else [(l, l + 1) for l in range(L)]

    def run(synced):
        ctx = B.D2OContext(B.make_config(n_layers=L, batch=B_, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=P,
                                         max_new_tokens=tokens + 3, rho=(small + large) / 2 / P, n_sink=1, window=8, min_budget=16))
        for l in range(L):
            ctx.d2o_layer_stats(l, Q[l], K[l])
        for l in range(L):                                                 # Eq. 5 weights exp(-F)
            ctx.density()[:, l] = 1.0 - torch.log(torch.tensor(large if l in big else small)).item()
        budgets = ctx.d2o_layer_budgets()
        assert all(bool((budgets[:, l] * row > 20e6).all()) == (l in big) for l in range(L))
        ctx.d2o_prefill_compress_layers(0, L, list(K), list(V))
        at = ctx._view(0).tau - ctx.state.data_ptr() + (L * B_ * hkv * 4 + 255) // 256 * 256      # the counters lie behind tau
        counters = ctx.state[at:at + L * B_ * hkv * 4].view(torch.int32).view(L, -1)
        out = torch.zeros_like(q)
        written = []
        for t in range(tokens):
            for l0, l1 in calls:
                ctx.d2o_decode_step(l0, l1, q[t, l0:l1], k[t, l0:l1], v[t, l0:l1], out[t, l0:l1])
                if synced:
                    torch.cuda.synchronize()
            written.append(counters.clone())
        torch.cuda.synchronize()
        assert ctx.d2o_get_stats().error_word == 0
        for t, c in enumerate(written):                                    # those of layer 5 may be written by the next token's first call
            assert bool((c[0] == t + 1).all()) and bool((c[3] == t + 1).all()) and bool((c[5] >= t).all())
        tabs = ctx.tables()
        state = [ctx.slice_state(l, b, h, tabs) for l in range(L) for b in range(B_) for h in range(hkv)]
        ctx.close()
        return out, state

    want, ws = run(True)
    for _ in range(2):
        got, gs = run(False)
        assert torch.equal(want.view(torch.uint8), got.view(torch.uint8))
        for a, b in zip(ws, gs):
            assert all(torch.equal(a[key].view(torch.uint8), b[key].view(torch.uint8)) for key in ("pos", "score", "rnorm", "K", "V"))


@pytest.mark.parametrize("n,G,P,d,dtype", [(8, 4, 900, 128, "bf16"), (64, 1, 500, 128, "f16"), (5, 2, 70, 64, "f32")])
def test_uncompressed_outputs_are_the_next_queries(cuda_device, n, G, P, d, dtype):
    L, td = 12, B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    g = torch.Generator(device=cuda_device).manual_seed(P)
    kc, vc = (torch.randn(L, n, P + 2, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    q = torch.randn(n, G, d, generator=g, device=cuda_device).to(td)
    k, v = (torch.randn(L, n, d, generator=g, device=cuda_device).to(td) for _ in range(2))

    def run(synced):
        kk, vv = kc.clone(), vc.clone()
        out = torch.zeros(L, n, G, d, dtype=td, device=cuda_device)
        torch.cuda.synchronize()
        for l in range(L):
            B.d2o_full_decode_step(kk[l], vv[l], P, q if l == 0 else out[l - 1], k[l], v[l], out[l])
            if synced:
                torch.cuda.synchronize()
        # the second token reads the row that the first one has just appended
        for l in range(L):
            B.d2o_full_decode_step(kk[l], vv[l], P + 1, out[l - 1], k[l], v[l], out[l])
            if synced:
                torch.cuda.synchronize()
        return out, kk, vv

    want = run(True)
    for _ in range(5):
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(want, run(False)))


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


def _appended_then_summed(cuda_device, dtype, d, n, P, sums):
    """An uncompressed step that appends a row to a cache, and at once the column sums with that cache's keys and values as keys
    and queries, on the same stream: the step's kernel lets the next ones start as its first act.  Bit for bit the result of the
    calls with a synchronisation in between."""
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    g = torch.Generator(device=cuda_device).manual_seed(P + d)
    kc, vc = (torch.randn(n, P, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    q = torch.randn(n, 1, d, generator=g, device=cuda_device).to(td)
    k, v = (3 * torch.randn(n, d, generator=g, device=cuda_device).to(td) for _ in range(2))
    out = torch.empty_like(q)

    def run(synced):
        kc[:, P - 1].zero_()                              # as it was before the step
        vc[:, P - 1].zero_()
        torch.cuda.synchronize()
        B.d2o_full_decode_step(kc, vc, P - 1, q, k, v, out)
        if synced:
            torch.cuda.synchronize()
        got = sums(vc.view(1, n, P, d), kc.view(1, n, P, d))
        torch.cuda.synchronize()
        return got

    want = run(True)
    for _ in range(10):
        assert torch.equal(want, run(False))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,P", [(2, 200), (8, 2000), (32, 2000)])
def test_fp32_column_sums_of_a_cache_that_is_being_appended_to(cuda_device, n, P, d):
    cs = torch.empty(1, n, P, device=cuda_device)
    density = torch.empty(1, n, dtype=torch.float64, device=cuda_device)

    def static(Q, K):
        B.d2o_layer_stats_static(Q, K, cs, density)
        return cs.clone()

    _appended_then_summed(cuda_device, "f32", d, n, P, static)


@pytest.mark.parametrize("dtype,d,n,P", [("f32", 64, 8, 2000), ("f32", 64, 2, 12001), ("f32", 128, 2, 12001), ("f16", 128, 8, 1000),
                                          ("bf16", 64, 2, 777), ("f16", 64, 64, 300)])
def test_column_sums_of_a_context_behind_an_appending_step(cuda_device, dtype, d, n, P):
    """Heads with and without room for their dot products, and the CUDA-core sweeps on 16-bit inputs."""
    ctx = B.D2OContext(B.make_config(n_layers=1, batch=1, n_q_heads=n, n_kv_heads=n, d_head=d, dtype=dtype, prompt_len=P,
                                     max_new_tokens=1, rho=0.5, n_sink=1, min_budget=8))
    ctx.d2o_set_tuning(stats_path=1)

    def stats(Q, K):
        ctx.d2o_layer_stats(0, Q, K)
        return ctx.colsum(0).clone()

    _appended_then_summed(cuda_device, dtype, d, n, P, stats)
    ctx.close()
