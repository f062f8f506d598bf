"""The fp32 emission layer at the edges of its tiles.  The tile a call takes follows from the number of samples it asks for, and
every result is the same chain of multiply-adds in all of them, so parts of a call equal the whole bit for bit; the oracle is
met at the fp32 path's 1e-5."""
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


# worker counts around the tiles of 16, 32 and 64 and around the row pitch, hidden widths that are not whole slabs of 16, sample counts around
# the tiles of 4 to 64, calls at the borders between the tiles (1776 of them: 12 for each of 148 SMs),
# and hidden widths up to the largest whose weights stay in shared memory (N <= 16: any, else 652) and beyond
@pytest.mark.parametrize("N,D,H,S", [(1, 4, 4, 7), (3, 4, 12, 9), (63, 4, 20, 33), (64, 4, 8, 9472), (65, 4, 36, 4737), (130, 8, 8, 3200),
                                     (257, 8, 24, 2049), (4096, 4, 16, 161),
                                     (16, 4, 32, 14201), (17, 4, 32, 7101), (33, 4, 28, 28417), (16, 4, 32, 113700), (15, 4, 664, 65), (9, 4, 668, 65),
                                     (32, 4, 620, 130), (40, 4, 624, 130), (16, 4, 1024, 14300), (17, 4, 652, 7200), (64, 4, 652, 3700),
                                     (33, 4, 656, 130), (64, 8, 128, 14201), (64, 4, 32, 18945), (128, 8, 128, 16384), (4096, 16, 592, 37)])
def test_every_tile_gives_the_same_draws(N, D, H, S):
    w = inputs.make_weights(N, D, H, seed=N, fan_in_ref=32)
    gpu = binding.Cutoff(N, D, H, 1, S, seed=5)
    orc = O.CutoffOracle(w, 1, S, seed=5)
    for load in range(2):                                  # weights loaded over others: the draws are the last ones'
        gpu.load_weights(w if load else inputs.make_weights(N, D, H, seed=N + 1, fan_in_ref=32))
    for x in inputs.make_trace(N, 3, seed=S, sigma=0.25):
        gpu.push(x)
        orc.push(x)
    x = gpu.debug_samples(0, S)
    for first, n in [(0, min(S, 5)), (S // 2, min(33, S - S // 2)), (S - 1, 1)]:
        assert np.array_equal(gpu.debug_samples(first, n), x[first:first + n])
    rows = np.unique(np.linspace(0, S - 1, 80).astype(int))
    ref = orc.samples(rows)
    assert np.max(np.abs(x[rows] - ref) / np.maximum(np.abs(ref), np.abs(ref).mean())) <= 1e-5
