"""The encoder's recurrences at hidden widths that the register-resident kernel does not serve, against the oracle: windows of one step
and longer."""
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


@pytest.mark.parametrize("H,lag", [(96, 0), (96, 20), (160, 3), (192, 6), (224, 1), (256, 2), (136, 4)])
def test_encoder_widths_meet_the_oracle(H, lag):
    N, D, S = 37, 8, 40
    w = inputs.make_weights(N, D, H, seed=H, fan_in_ref=32)
    gpu = binding.Cutoff(N, D, H, lag, S, seed=3)
    gpu.load_weights(w)
    orc = O.CutoffOracle(w, lag, S, seed=3)
    for x in inputs.make_trace(N, lag + 4, seed=5, sigma=0.25):
        gpu.push(x)
        orc.push(x)
    x, ref = gpu.debug_samples(0, S), orc.samples(np.arange(S))
    assert np.max(np.abs(x - ref) / np.maximum(np.abs(ref), np.abs(ref).mean())) <= 1e-5

