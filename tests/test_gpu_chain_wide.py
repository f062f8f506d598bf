"""The chain with D lanes per sample, taken by decisions of few samples: edges of its batches and of the rule that chooses it."""
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


# every D; hidden widths with idle lanes (H < 4 D) and with a ragged last block; sample counts around a warp's 32 / D; windows of
# one step and long ones; both precisions; one and two samples per lane; the largest decision that takes either form and the
# smallest that does not (148 SMs)
@pytest.mark.parametrize("N,D,H,lag,S,prec", [(5, 4, 4, 0, 1, 0), (17, 4, 36, 3, 9, 0), (9, 8, 8, 20, 5, 0), (40, 8, 72, 20, 131, 0), (33, 16, 48, 1, 3, 0),
                                              (64, 16, 256, 4, 77, 1), (20, 32, 32, 0, 2, 0), (50, 32, 160, 6, 65, 2), (16, 16, 64, 2, 2368, 1),
                                              (16, 16, 64, 2, 2369, 1), (16, 8, 32, 2, 7104, 0), (16, 8, 32, 2, 7109, 0),
                                              (16, 8, 32, 2, 23680, 0), (16, 8, 32, 2, 23689, 0), (16, 4, 32, 1, 20001, 0),
                                              (33, 16, 48, 1, 4001, 0), (16, 32, 32, 1, 1999, 0), (16, 32, 32, 1, 2400, 0)])
def test_wide_chain_meets_the_oracle(N, D, H, lag, S, prec):
    w = inputs.make_weights(N, D, H, seed=N + D, fan_in_ref=32, bf16=(prec == 2))
    gpu = binding.Cutoff(N, D, H, lag, S, precision=prec, seed=3)
    gpu.load_weights(w)
    orc = O.CutoffOracle(w, lag, S, seed=3)
    for x in inputs.make_trace(N, lag + 3, seed=S, sigma=0.25):
        gpu.push(x)
        orc.push(x)
    x = gpu.debug_samples(0, S)
    rows = np.unique(np.linspace(0, S - 1, 100).astype(int))
    ref = orc.samples(rows)
    tol = 1e-5 if prec == 0 else 2e-3
    assert np.max(np.abs(x[rows] - ref) / np.maximum(np.abs(ref), np.abs(ref).mean())) <= tol
    first, n = S // 3, min(7, S - S // 3)
    assert np.array_equal(gpu.debug_samples(first, n), x[first:first + n])


def test_shards_of_a_decision_take_the_same_chain():
    # 8192 samples in all: the whole decision does not take this chain, so its shards of 1024 must not either
    N, D, H, lag, S = 24, 16, 64, 2, 8192
    w = inputs.make_weights(N, D, H, seed=1, fan_in_ref=32)
    trace = inputs.make_trace(N, lag + 2, seed=2, sigma=0.25)
    whole = binding.Cutoff(N, D, H, lag, S, precision=1, seed=3)
    part = binding.Cutoff(N, D, H, lag, S // 8, precision=1, seed=3, sample_offset=3 * S // 8, total_samples=S)
    for g in (whole, part):
        g.load_weights(w)
        for x in trace:
            g.push(x)
    assert np.array_equal(part.debug_samples(0, S // 8), whole.debug_samples(3 * S // 8, S // 8))
