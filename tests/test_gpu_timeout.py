"""Failure detection: a device-side wait that runs out is reported, nothing hangs, nothing traps.

The decode kernel waits for stages of cache rows that its copy engine delivers.  The test knob
d2o_set_fault_injection makes one stage never arrive and shortens the wait limit to two
milliseconds: the kernel must come back on its own, leave the slice untouched, and report
D2O_ERR_TIMEOUT through d2o_get_stats; later steps on the same context do nothing; the CUDA context
stays usable for a fresh library context.
"""
import dataclasses
import time

import pytest
import torch

from paper_2406_13035_b200 import binding as B
from paper_2406_13035_b200 import workloads as W

from parity import assert_report, make_ctx, run_parity

pytestmark = pytest.mark.gpu

D2O_ERR_STATE = 4
D2O_ERR_TIMEOUT = 6


def _state(ctx, wl):
    tabs = ctx.tables()
    return [ctx.slice_state(0, 0, h, tabs) for h in range(wl.n_kv_heads)]


def _same(a, b):
    return all(x["len"] == y["len"] and x["tau"] == y["tau"] and torch.equal(x["pos"], y["pos"]) and
               torch.equal(x["score"], y["score"]) and torch.equal(x["K"], y["K"]) and torch.equal(x["V"], y["V"])
               for x, y in zip(a, b))


@pytest.mark.parametrize("name", ["cfg0", "cfg2"])
def test_decode_wait_that_runs_out_is_reported(cuda_device, name):
    from paper_2406_13035_b200 import build
    build.build_library()
    B.load_library()
    base = W.CONFIGS["cfg0"] if name == "cfg0" else W.twin("cfg2")
    # caches of ~200 rows: several stages per pass, so that stage 1 belongs to the key pass
    wl = dataclasses.replace(base, prompt_len=512, decode_steps=4, n_layers=1, batch=1, max_budget=0, rho=0.4)
    ctx = make_ctx(wl)
    s = W.LayerStream(wl, 0, "cuda:0")
    Q, K, V = s.prompt()
    ctx.d2o_layer_stats(0, Q, K)
    ctx.d2o_layer_budgets()
    ctx.d2o_prefill_compress(0, K, V)
    q, k, v = s.decode()
    out = torch.zeros_like(q)
    ctx.d2o_decode_step(0, 1, q, k, v, out)                      # an ordinary step first
    torch.cuda.synchronize()
    assert ctx.d2o_get_stats().error_word == 0
    before = _state(ctx, wl)
    # stage 1 of every slice never arrives; a wait gives up after 2 ms
    ctx.d2o_set_fault_injection(wait_limit_us=2000, producer_stop_stage=1)
    q, k, v = s.decode()
    t0 = time.perf_counter()
    ctx.d2o_decode_step(0, 1, q, k, v, out)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    st = ctx.d2o_get_stats()
    assert st.error_word == D2O_ERR_TIMEOUT, (st.error_word, hex(st.error_detail))
    assert dt < 2.0, f"the step took {dt:.3f} s"
    assert _same(before, _state(ctx, wl))                        # the wait ran out in the key pass: nothing was written
    # later steps on this context do nothing and return at once, with or without the knob
    ctx.d2o_set_fault_injection(0, -1)
    q, k, v = s.decode()
    t0 = time.perf_counter()
    ctx.d2o_decode_step(0, 1, q, k, v, out)
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 0.5
    assert ctx.d2o_get_stats().error_word == D2O_ERR_TIMEOUT
    assert _same(before, _state(ctx, wl))
    ctx.close()
    # the CUDA context is intact: a fresh library context passes an ordinary parity run
    small = dataclasses.replace(W.CONFIGS["cfg0"], prompt_len=128, decode_steps=2)
    rep = run_parity(small)
    assert_report(rep, small.dtype)


@pytest.mark.parametrize("P,rho,hq,hkv,d,dtype,stage", [
    (400, 0.5, 8, 8, 64, "f32", 4),             # 200 rows on two CTAs: the first copy of values
    (640, 0.505, 8, 2, 128, "bf16", 3),         # 323 rows on four
    (640, 0.505, 8, 2, 128, "bf16", 5),         # the last copy of values
    (1900, 0.9, 2, 1, 128, "f32", 7)])          # 1710 rows on eight
def test_decode_cluster_whose_values_do_not_arrive(cuda_device, P, rho, hq, hkv, d, dtype, stage):
    """The CTAs of a cluster leave together, after the stores that they send one another (outputs and the new token's entry)
    have landed; nothing of the slice is written, and later steps, which leave at the first barrier, do nothing either."""
    wl = dataclasses.replace(W.CONFIGS["cfg0"], n_layers=1, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype,
                             prompt_len=P, rho=rho, decode_steps=8, min_budget=8, max_budget=0)
    ctx = make_ctx(wl)
    s = W.LayerStream(wl, 0, "cuda:0")
    Q, K, V = s.prompt()
    ctx.d2o_layer_stats(0, Q, K)
    ctx.d2o_layer_budgets()
    ctx.d2o_prefill_compress(0, K, V)
    q, k, v = s.decode()
    out = torch.zeros_like(q)
    ctx.d2o_decode_step(0, 1, q, k, v, out)
    before, first = _state(ctx, wl), out.clone()
    assert ctx.d2o_get_stats().error_word == 0
    ctx.d2o_set_fault_injection(wait_limit_us=2000, producer_stop_stage=stage)
    for _ in range(4):                                           # the step that runs out of time, then steps that find the error
        t0 = time.perf_counter()
        ctx.d2o_decode_step(0, 1, q, k, v, out)
        torch.cuda.synchronize()
        assert time.perf_counter() - t0 < 0.5
        assert ctx.d2o_get_stats().error_word == D2O_ERR_TIMEOUT
        assert _same(before, _state(ctx, wl)) and torch.equal(out, first)
    ctx.close()


@pytest.mark.parametrize("P,rho,hq,hkv,d,dtype", [(400, 0.5, 8, 8, 64, "f32"), (640, 0.505, 8, 2, 128, "bf16")])
def test_layers_behind_one_that_ran_out_of_time(cuda_device, P, rho, hq, hkv, d, dtype):
    """The next layers' clusters are already resident when a layer's wait runs out; they too do nothing."""
    wl = dataclasses.replace(W.CONFIGS["cfg0"], n_layers=3, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype,
                             prompt_len=P, rho=rho, decode_steps=8, min_budget=8, max_budget=0)
    ctx = make_ctx(wl)
    streams = [W.LayerStream(wl, l, "cuda:0") for l in range(3)]
    kv = []
    for l, s in enumerate(streams):
        Q, K, V = s.prompt()
        ctx.d2o_layer_stats(l, Q, K)
        kv.append((K, V))
    ctx.d2o_layer_budgets()
    for l in range(3):
        ctx.d2o_prefill_compress(l, *kv[l])
    first = [s.decode() for s in streams]
    second = [s.decode() for s in streams]
    out = [torch.zeros_like(q) for q, _, _ in first]
    for l in range(3):
        ctx.d2o_decode_step(l, l + 1, *first[l], out[l])
    torch.cuda.synchronize()
    assert ctx.d2o_get_stats().error_word == 0

    def state():
        tabs = ctx.tables()
        return [ctx.slice_state(l, 0, h, tabs) for l in range(3) for h in range(hkv)]

    before, first_out = state(), [o.clone() for o in out]
    ctx.d2o_set_fault_injection(wait_limit_us=2000, producer_stop_stage=1)
    ctx.d2o_decode_step(0, 1, *second[0], out[0])
    ctx.d2o_set_fault_injection(0, -1)
    for l in (1, 2):
        ctx.d2o_decode_step(l, l + 1, *second[l], out[l])
    torch.cuda.synchronize()
    assert ctx.d2o_get_stats().error_word == D2O_ERR_TIMEOUT
    assert _same(before, state()) and all(torch.equal(a, b) for a, b in zip(first_out, out))
    ctx.close()


@pytest.mark.parametrize("word,taken", [(D2O_ERR_STATE, True), (D2O_ERR_TIMEOUT, False)])
@pytest.mark.parametrize("hq,hkv,d,dtype", [(8, 8, 64, "f32"), (32, 8, 128, "bf16")])
def test_error_recorded_while_a_step_waits(cuda_device, hq, hkv, d, dtype, word, taken):
    """A step on clusters that is resident and waits for the kernel ahead of it when an error is recorded: one that concerns a single
    slice (its token was dropped) does not stop it, a wait that ran out does."""
    wl = dataclasses.replace(W.CONFIGS["cfg0"], n_layers=2, batch=1, n_q_heads=hq, n_kv_heads=hkv, d_head=d, dtype=dtype, prompt_len=300,
                             rho=0.4, decode_steps=8, min_budget=8, max_budget=0)
    ctx = make_ctx(wl)
    streams = [W.LayerStream(wl, l, "cuda:0") for l in range(2)]
    Q, K, V = zip(*[s.prompt() for s in streams])
    ctx.d2o_layer_stats_layers(0, 2, Q, K)
    ctx.d2o_layer_budgets()
    ctx.d2o_prefill_compress_layers(0, 2, K, V)
    for _ in range(2):
        for l in range(2):
            q, k, v = streams[l].decode()
            out = torch.empty_like(q)
            ctx.d2o_decode_step(l, l + 1, q, k, v, out)
    q, k, v = streams[0].decode()
    # eight CTAs that take milliseconds over a long cache, and let the step move in at once
    kc, vc = (torch.zeros(1, 1 << 20, 128, device=cuda_device) for _ in range(2))
    x = torch.zeros(1, 1, 128, device=cuda_device)
    error = torch.tensor([word], dtype=torch.int32).pin_memory()
    at = ctx.state[ctx._state_off:ctx._state_off + 4].view(torch.int32)
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    assert ctx.d2o_get_stats().error_word == 0
    before = ctx.d2o_get_stats().decode_steps
    torch.cuda.synchronize()
    B.d2o_full_decode_step(kc, vc, (1 << 20) - 1, x, x[0], x[0], torch.empty_like(x))
    ctx.d2o_decode_step(0, 1, q, k, v, out)
    done.record()
    time.sleep(2e-4)
    with torch.cuda.stream(side):
        at.copy_(error, non_blocking=True)
    side.synchronize()
    assert not done.query()                                      # the kernel ahead was still running
    torch.cuda.synchronize()
    assert ctx.d2o_get_stats().decode_steps - before == (hkv if taken else 0)
    ctx.close()


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f16", 64)])
@pytest.mark.parametrize("P,hq,stage", [(1025, 2, 0), (1025, 2, 1), (1025, 2, 3), (700, 64, 5), (2000, 40, 9)])
def test_column_sums_whose_tiles_do_not_arrive(cuda_device, dtype, d, P, hq, stage):
    """Fewer items than SMs and more (those that a CTA takes behind its first one, and those that nobody takes any more), a
    wait that runs out in the first item or later.  Every column sum that the missing tiles could have entered is NaN; a call
    without the knob afterwards computes everything."""
    g = torch.Generator(device=cuda_device).manual_seed(P)
    td = B.TORCH_DTYPE[B.DTYPE_CODE[dtype]]
    Q = torch.randn(1, hq, P, d, generator=g, device=cuda_device).to(td)
    K = torch.randn(1, hq, P, d, generator=g, device=cuda_device).to(td)
    make = lambda: B.D2OContext(B.make_config(n_layers=1, batch=1, n_q_heads=hq, n_kv_heads=hq, d_head=d, dtype=dtype,
                                              prompt_len=P, max_new_tokens=2, rho=0.5, n_sink=1, min_budget=8))
    ctx, other = make(), make()
    other.d2o_layer_stats(0, Q, K)
    ctx.d2o_set_fault_injection(wait_limit_us=2000, producer_stop_stage=stage)
    t0 = time.perf_counter()
    ctx.d2o_layer_stats(0, Q, K)
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 1.0
    assert ctx.d2o_get_stats().error_word == D2O_ERR_TIMEOUT
    cs = ctx.colsum(0)
    # the last rows' normalisers take every tile of the keys; they enter every column of their head
    assert torch.isnan(cs).all()
    ctx.d2o_set_fault_injection(0, -1)
    ctx.d2o_layer_stats(0, Q, K)
    assert torch.equal(ctx.colsum(0), other.colsum(0))
    ctx.close()
    other.close()
