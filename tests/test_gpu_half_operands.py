"""The emission products on half-precision operands with a power of two per row taken out: what must hold exactly.

Powers of two move through tf32 rounding, the scaling of a row, the products and their fp32 sums without rounding, so a
hidden layer scaled by 2^a against output weights scaled by 2^-a, and a worker's mean row scaled by 2^k, change results by
exactly those powers: the tolerance is zero.  The oracle is met at the tensor-core path's 2e-3."""
import numpy as np
import pytest

from oracle import cutoff_oracle as O
from paper_1803_04209_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "these tests need a GPU"
    build.build()
    return binding.load_library()


def samples(w, trace, D, H, lag, S, prec, literal, parts=False):
    gpu = binding.Cutoff(trace.shape[1], D, H, lag, S, precision=prec, seed=77, flags=binding.FLAG_LITERAL if literal else 0)
    gpu.load_weights(w)
    for x in trace:
        gpu.push(x)
    out = gpu.debug_samples(0, S)
    if parts:                                            # a few rows by themselves: other tiles, other blocks
        assert np.array_equal(gpu.debug_samples(S // 3, min(9, S - S // 3)), out[S // 3: S // 3 + 9])
    return out


# row pitches that need padding (H = 36, 72, 264), weights that stay in shared memory (H <= 256) and that do not, chains on
# and off the tensor cores, one worker, the edges of a worker tile, blocks that go from one worker tile to the next
@pytest.mark.parametrize("N,D,H,S,prec", [(1, 4, 36, 130, 1), (127, 8, 72, 129, 2), (129, 16, 128, 300, 1), (300, 16, 256, 257, 1),
                                          (40, 8, 264, 200, 1), (257, 32, 320, 140, 2), (700, 16, 64, 4000, 1), (4096, 32, 256, 700, 2)])
@pytest.mark.parametrize("literal", [False, True])
def test_powers_of_two_pass_through_exactly(N, D, H, S, prec, literal):
    lag = 1
    make = inputs.make_weights_literal if literal else inputs.make_weights
    w = make(N, D, H, seed=N + H, fan_in_ref=32, bf16=(prec == 2))
    trace = inputs.make_trace(N, lag + 2, seed=S, sigma=0.25)
    x = samples(w, trace, D, H, lag, S, prec, literal, parts=True)

    orc = O.CutoffOracle(w, lag, S, seed=77)
    for t in trace:
        orc.push(t)
    rows = np.unique(np.linspace(0, S - 1, 60).astype(int))
    ref = orc.samples(rows)
    assert np.max(np.abs(x[rows] - ref) / np.maximum(np.abs(ref), np.abs(ref).mean())) <= 2e-3

    hidden, out = (("Wi1", "bi1"), ("Wi2",)) if literal else (("W3", "b3"), ("W4",))
    for a in (-30, 30):
        v = {k: t.copy() for k, t in w.items()}
        for k in hidden:
            v[k] *= np.float32(2.0 ** a)
        for k in out:
            v[k] *= np.float32(2.0 ** -a)
        if literal:                                      # and the hidden layer of the scale the other way
            for k in ("Wj1", "bj1"):
                v[k] *= np.float32(2.0 ** -a)
            v["Wj2"] *= np.float32(2.0 ** a)
        assert np.array_equal(samples(v, trace, D, H, lag, S, prec, literal), x), a

    # without noise a worker's sample is its mean row alone, whatever the other rows' sizes
    quiet = {k: t.copy() for k, t in w.items()}
    if literal:
        quiet["bj2"][:] = -300.0
    else:
        quiet["b4"][N:] = -400.0
    x0 = samples(quiet, trace, D, H, lag, S, prec, literal)
    power = np.random.default_rng(N).integers(-20, 21, N)
    two = (np.float32(2.0) ** power).astype(np.float32)
    mean, bias = ("Wi2", "bi2") if literal else ("W4", "b4")
    quiet[mean][:N] *= two[:, None]
    quiet[bias][:N] *= two
    if literal:                                          # M = Wj1 Wi2 would mix the rows
        quiet["Wj1"][:] = 0.0
    assert np.array_equal(samples(quiet, trace, D, H, lag, S, prec, literal), x0 * two)


@pytest.mark.parametrize("N,D,H,S,literal", [(40, 16, 64, 2500, False), (40, 16, 64, 300, False), (40, 8, 64, 300, False), (40, 32, 64, 3000, False),
                                             (40, 16, 64, 300, True)])
def test_a_captured_graph_follows_reloaded_weights(N, D, H, S, literal):
    # the bound a hidden vector is scaled by belongs to the weights, not to the graph: reloaded ones may be far larger
    make = inputs.make_weights_literal if literal else inputs.make_weights
    w = make(N, D, H, seed=1, fan_in_ref=32)
    big = {k: t.copy() for k, t in w.items()}
    hidden, out = (("Wi1", "bi1"), "Wi2") if literal else (("W3", "b3"), "W4")
    for k in hidden:
        big[k] *= np.float32(2.0 ** 24)
    big[out] *= np.float32(2.0 ** -24)
    trace = inputs.make_trace(N, 6, seed=2, sigma=0.25)
    flags = binding.FLAG_LITERAL if literal else 0
    stats = []
    for graph in (binding.FLAG_GRAPH, 0):
        gpu = binding.Cutoff(N, D, H, 1, S, precision=1, seed=77, flags=flags | graph)
        gpu.load_weights(w)
        for i, x in enumerate(trace):
            if i == 4:
                gpu.load_weights(big)
            gpu.step(x)
        stats.append(gpu.get_stats()[0])
    assert np.all(np.isfinite(stats[0])) and np.array_equal(stats[0], stats[1])


# A unit that is switched off by its bias contributes nothing, and nothing about the others may depend on how far off it is:
# the same samples to the last bit.  Chains: wide, resident, tensor cores with D = 16 and 32; literal: the hidden layer of the scale.
@pytest.mark.parametrize("N,D,H,S,literal", [(40, 8, 72, 300, False), (40, 4, 32, 60000, False), (300, 16, 128, 3000, False), (300, 32, 256, 3000, False),
                                             (300, 16, 128, 300, True), (40, 8, 72, 300, True)])
def test_units_that_are_switched_off_cost_the_others_nothing(N, D, H, S, literal):
    make = inputs.make_weights_literal if literal else inputs.make_weights
    w = make(N, D, H, seed=N + H, fan_in_ref=32)
    trace = inputs.make_trace(N, 3, seed=S, sigma=0.25)
    hidden, bias = ("Wj1", "bj1") if literal else ("W3", "b3")
    w[hidden][::5] = 0.0
    out = []
    for off in (-1.0, -2.0 ** 20, -2.0 ** 34, -2.0 ** 100):
        w[bias][::5] = off
        out.append(samples(w, trace, D, H, 1, min(S, 3000), 1, literal) if S <= 3000 else _head(w, trace, D, H, S))
    for x in out[1:]:
        assert np.array_equal(x, out[0])


def _head(w, trace, D, H, S):
    gpu = binding.Cutoff(trace.shape[1], D, H, 1, S, precision=1, seed=77)
    gpu.load_weights(w)
    for x in trace:
        gpu.push(x)
    return gpu.debug_samples(S // 2, 500)


# rows of weights whose size lies near either end of the fp32 range, up to results of 2^125
@pytest.mark.parametrize("N,D,H,S", [(40, 8, 72, 300), (300, 16, 128, 3000)])
@pytest.mark.parametrize("power", [-100, 100, 121])
def test_rows_of_weights_near_the_ends_of_the_range(N, D, H, S, power):
    w = inputs.make_weights(N, D, H, seed=N + H, fan_in_ref=32)
    w["b4"][N:] = -400.0                                 # no noise: a worker's sample is its mean row alone
    trace = inputs.make_trace(N, 3, seed=S, sigma=0.25)
    x = samples(w, trace, D, H, 1, S, 1, False)
    assert np.abs(x).max() < 8
    two = np.float32(2.0 ** power)
    w["W4"][:N:2] *= two
    w["b4"][:N:2] *= two
    x[:, ::2] *= two
    assert np.array_equal(samples(w, trace, D, H, 1, S, 1, False), x)
