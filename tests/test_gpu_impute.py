"""Imputation of censored workers, spread over several CTAs: every replacement is the worker's first draw above the threshold."""
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


# fewer workers than CTAs, one more than a multiple of them, every worker of one CTA censored, the most workers; columns
# shorter than the 256 draws in flight and several times longer
@pytest.mark.parametrize("N,S,keep", [(2, 40, [0]), (5, 300, [1, 4]), (17, 1000, [3]), (33, 256, list(range(1, 33, 2))), (4096, 257, [7, 4095])])
def test_replacements_are_the_gpus_own_draws(N, S, keep):
    seed = 11
    gpu = binding.Cutoff(N, 4, 16, 1, S, seed=seed)
    gpu.load_weights(inputs.make_weights(N, 4, 16, seed=N, fan_in_ref=32))
    trace = inputs.make_trace(N, 4, seed=S, sigma=0.3)
    for x in trace[:3]:
        gpu.push(x)
    scale = np.float32(2.0 * trace[:2].astype(np.float64).mean())
    draws = gpu.debug_samples(0, S) * scale
    gpu.predict()
    observed = np.sort(draws, axis=0)[S // 2].astype(np.float32).clip(0.05)      # about half of a column lies above its middle
    censored = np.ones(N, dtype=bool)
    censored[keep] = False
    gpu.push(np.where(censored, np.nan, observed).astype(np.float32), censored)
    got = gpu.debug_window()[-1]
    threshold = observed[~censored].max()
    assert np.array_equal(got[~censored], observed[~censored])
    for j in np.flatnonzero(censored):
        start = int(O.philox4x32_10(int(j), 0, O.STREAM_IMPUTE, 1, seed & 0xFFFFFFFF, seed >> 32)[0]) % S
        column = np.roll(draws[:, j], -start)
        if np.min(np.abs(column - threshold)) <= 1e-6 * threshold:
            continue                                             # the scale's last bit decides
        hits = np.flatnonzero(column > threshold)
        assert abs(got[j] - (column[hits[0]] if hits.size else threshold)) <= 1e-6 * threshold
