"""Orders of calls in which one call's work is still under way when the next is made."""
import numpy as np
import pytest

from paper_1803_04209_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "these tests need a GPU"
    build.build()
    return binding.load_library()


def _running(N, D, H, lag, S, precision=0, flags=0):
    ctx = binding.Cutoff(N, D, H, lag, S, precision=precision, seed=5, flags=flags)
    ctx.load_weights(inputs.make_weights(N, D, H, seed=N, fan_in_ref=32))
    trace = inputs.make_trace(N, lag + 6, seed=S, sigma=0.3)
    for x in trace[: lag + 1]:
        ctx.push(x)
    return ctx, trace[lag + 1:]


@pytest.mark.parametrize("N,S", [(16, 1024), (1025, 300)])
def test_a_bad_push_behind_a_decision_does_not_take_the_decision_away(N, S):
    import torch
    ctx, trace = _running(N, 4, 32, 1, S)
    want = ctx.predict()
    stats = ctx.get_stats()
    ctx.reset()
    for x in inputs.make_trace(N, 7, seed=S, sigma=0.3)[:2]:
        ctx.push(x)
    bad = torch.from_numpy(trace[0]).cuda()
    bad[N // 2] = float("nan")
    ctx.predict_async()
    ctx.push_async(bad)
    assert ctx.fetch() == want
    assert all(np.array_equal(a, b) for a, b in zip(ctx.get_stats(), stats))
    ctx.predict_async()                                  # the bad vector is reported by the next decision ...
    with pytest.raises(binding.CutoffError) as e:
        ctx.fetch()
    assert e.value.code == binding.ERR_BAD_VALUE
    window = ctx.debug_window()                          # ... and never entered the window
    assert np.array_equal(window, inputs.make_trace(N, 7, seed=S, sigma=0.3)[:2])
    assert ctx.predict()[0] >= 0


def test_a_host_push_keeps_its_run_times_when_a_replayed_step_follows():
    # both land in one buffer on the host: the step may not fill it before the push's kernel has read it
    N, lag = 4096, 3
    ctx, trace = _running(N, 4, 32, lag, 64, flags=binding.FLAG_GRAPH)
    lib, c = binding.load_library(), binding.C.c_int32(0)
    ctx.predict()
    ctx.step(trace[0])                                   # captured here
    window = list(ctx.debug_window())
    rng = np.random.default_rng(0)
    for _ in range(200):
        first, second = rng.uniform(0.5, 2.0, (2, N)).astype(np.float32)
        a, b = first.ctypes.data, second.ctypes.data
        push, step = lib.cutoff_push, lib.cutoff_step
        assert push(ctx._h, a, 0, None) == 0 and step(ctx._h, b, binding.C.byref(c)) == 0
        window = (window + [first, second])[-(lag + 1):]
        assert np.array_equal(ctx.debug_window(), np.stack(window))
