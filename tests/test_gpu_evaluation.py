"""The library's evaluation of cutoff rules on recorded traces against the oracle's (Sections 3, 3.1.1, 4.1).

Throughputs are ratios of an integer and an observed fp32 run-time, formed in double on both sides, so the
hindsight cutoffs must agree exactly and the throughputs to fp32 rounding.  The "order" rule goes through running
sums and a normal quantile, which the two sides round differently in the last bits of a double: its cutoffs must
agree unless two cutoffs tie to within 1e-9.
"""
import numpy as np
import pytest

from oracle import evaluation as E
from paper_1803_04209_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "these tests need a GPU"
    build.build()
    return binding.load_library()


def _trace(N, T, seed):
    return inputs.make_trace(N, T, seed=seed, sigma=0.3, groups=min(4, N), stay=0.85, slowdown=2.0,
                             straggler_p=0.03, straggler_scale=1.5)


@pytest.mark.parametrize("N,T", [(1, 5), (2, 9), (16, 40), (33, 17), (158, 64), (1024, 50), (1025, 9), (2175, 12), (4096, 10)])
def test_eval_trace_matches_the_oracle(N, T):
    import torch
    trace = _trace(N, T, seed=N + T)
    trace[T // 2] = trace[T // 2, 0]                                   # one step of equal run-times
    if N >= 4:
        trace[1] = (np.arange(N) + 1) * np.float32(0.125)              # Omega constant: the tie goes to c = N
    rng = np.random.default_rng(N)
    rules = np.stack([np.full(T, N), np.full(T, max(1, N // 2)), rng.integers(1, N + 1, size=T),
                      np.array([E.hindsight_best(row)[0] for row in trace])]).astype(np.int32)
    got = binding.eval_trace(torch.from_numpy(trace).cuda(), torch.from_numpy(rules).cuda())
    want = E.evaluate(trace, {f"r{m}": rules[m] for m in range(rules.shape[0])})
    assert np.array_equal(got["best_c"].cpu().numpy(), want["best_c"])
    assert np.allclose(got["best"].cpu().numpy(), want["best"], rtol=1e-6, atol=0)
    assert np.allclose(got["all"].cpu().numpy(), want["all"], rtol=1e-6, atol=0)
    for m in range(rules.shape[0]):
        assert np.allclose(got["achieved"][m].cpu().numpy(), want[f"r{m}"], rtol=1e-6, atol=0)
        assert np.array_equal(got["step_time"][m].cpu().numpy(), want[f"r{m}_time"].astype(np.float32))
    assert np.array_equal(got["achieved"][3].cpu().numpy(), got["best"].cpu().numpy())   # the hindsight rule attains the maximum
    assert int(got["static_c"].item()) == E.best_static_cutoff(trace)
    # a padded leading dimension and no rules at all
    padded = torch.zeros((T, N + 5), dtype=torch.float32, device="cuda")
    padded[:, :N] = torch.from_numpy(trace).cuda()
    bare = binding.eval_trace(padded[:, :N], None, want_static=False)
    assert np.array_equal(bare["best_c"].cpu().numpy(), want["best_c"])


@pytest.mark.parametrize("N,T", [(1, 4), (24, 30), (158, 100), (1024, 60), (4096, 8)])
def test_order_baseline_matches_the_oracle(N, T):
    import torch
    trace = _trace(N, T, seed=7 * N + T)
    got = binding.order_baseline(torch.from_numpy(trace).cuda()).cpu().numpy()
    want = E.order_cutoffs(trace)
    assert got[0] == N
    x = trace.astype(np.float64)
    for t in np.flatnonzero(got != want):
        seen = x[:t].reshape(-1)
        e = E.elfving_expected(N, float(seen.mean()), float(seen.std()))
        om_got, om_want = got[t] / e[got[t] - 1], want[t] / e[want[t] - 1]
        assert abs(om_got - om_want) <= 1e-9 * abs(om_want), f"step {t}: cutoff {got[t]} != oracle {want[t]}"
    assert np.mean(got == want) >= 0.9


def test_eval_trace_rejects_bad_arguments():
    import torch
    lib = binding.load_library()
    t = torch.ones((3, 8), dtype=torch.float32, device="cuda")
    o = torch.zeros(3, dtype=torch.float32, device="cuda")
    oi = torch.zeros(3, dtype=torch.int32, device="cuda")
    assert lib.cutoff_eval_trace(0, None, 3, 8, 8, None, 0, oi.data_ptr(), o.data_ptr(), o.data_ptr(), None, None, None, None) == binding.ERR_BAD_ARG
    assert lib.cutoff_eval_trace(0, t.data_ptr(), 3, 4097, 4097, None, 0, oi.data_ptr(), o.data_ptr(), o.data_ptr(), None, None, None, None) == binding.ERR_BAD_ARG
    assert lib.cutoff_eval_trace(0, t.data_ptr(), 3, 8, 8, None, 1, oi.data_ptr(), o.data_ptr(), o.data_ptr(), None, None, None, None) == binding.ERR_BAD_ARG
    assert lib.cutoff_order_baseline(0, t.data_ptr(), 0, 8, 8, oi.data_ptr(), None) == binding.ERR_BAD_ARG


# running moments are scanned 1024 steps at a time, a warp at a time; the moments kernel takes 8 steps per CTA
@pytest.mark.parametrize("N,T", [(24, 1), (7, 33), (5, 1024), (5, 1025), (6, 2100)])
def test_order_baseline_over_long_traces(N, T):
    import torch
    trace = _trace(N, T, seed=N + 3 * T)
    got = binding.order_baseline(torch.from_numpy(trace).cuda()).cpu().numpy()
    x = trace.astype(np.float64)
    s1, s2 = np.cumsum(x.sum(1)), np.cumsum((x * x).sum(1))
    assert got[0] == N
    for t in range(1, T):
        mu, n = s1[t - 1] / (t * N), t * N
        e = E.elfving_expected(N, float(mu), float(np.sqrt(max(s2[t - 1] / n - mu * mu, 0.0))))
        want = E.cutoff_from_expected(e)
        # moments differ by the order of a sum in double: 1e-12 of the throughput at most
        assert got[t] == want or abs(got[t] / e[got[t] - 1] - want / e[want - 1]) <= 1e-9 * abs(want / e[want - 1]), t


def test_calls_from_several_threads_and_streams_do_not_share_scratch():
    import threading
    import torch
    cases = [(_trace(N, T, seed=N), torch.cuda.Stream()) for N, T in ((40, 300), (700, 80), (1500, 20), (64, 500))]
    wrong = []

    def work(trace, stream):
        dev = torch.from_numpy(trace).cuda()
        torch.cuda.synchronize()
        want_c, want_order = E.best_static_cutoff(trace), None
        with torch.cuda.stream(stream):
            for _ in range(5):
                c = int(binding.eval_trace(dev, None, stream=stream.cuda_stream)["static_c"].item())
                order = binding.order_baseline(dev, stream=stream.cuda_stream).cpu().numpy()
                want_order = order if want_order is None else want_order
                if c != want_c or not np.array_equal(order, want_order):
                    wrong.append((trace.shape, c, want_c))

    threads = [threading.Thread(target=work, args=c) for c in cases]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("N,T,outlier", [(24, 80, 1e15), (158, 40, 1e18), (5, 1100, 1e12)])
def test_order_baseline_does_not_see_the_step_it_decides(N, T, outlier):
    # a step's own run-times, however far out, must not reach its own moments, not even as a rounding error.  Moments are sums
    # in double whose order differs between the two sides: 1e-12 of the throughput at most
    import torch
    trace = _trace(N, T, seed=N + T)
    at = T - T // 4
    trace[at] = np.float32(outlier)
    got = binding.order_baseline(torch.from_numpy(trace).cuda()).cpu().numpy()
    x = trace.astype(np.float64)
    for t in range(1, at + 1):
        mu = float(x[:t].mean())
        e = E.elfving_expected(N, mu, float(np.sqrt(max(float((x[:t] * x[:t]).mean()) - mu * mu, 0.0))))
        want = E.cutoff_from_expected(e)
        assert got[t] == want or abs(got[t] / e[got[t] - 1] - want / e[want - 1]) <= 1e-9 * abs(want / e[want - 1]), t
