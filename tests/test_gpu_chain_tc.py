"""The chain on tensor cores: latent size 16 with every hidden width, latent size 32 with widths that fill and split blocks, windows of one step and longer, sample counts at the edges of its
tiles (64 samples, 128 samples with 16 or 8 warps) and of the rules that choose between them, against the oracle."""
import numpy as np
import pytest

from oracle import cutoff_oracle as O
from paper_1803_04209_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu

SMS = 148


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "these tests need a GPU"
    build.build()
    return binding.load_library()


# the compact model takes this chain from 2369 samples on, the literal one always
@pytest.mark.parametrize("D", [16, 32])
@pytest.mark.parametrize("H,lag,S,literal", [(64, 0, 2369, False), (128, 1, 2400, False), (192, 2, 64 * SMS, False), (256, 4, 64 * SMS + 1, False),
                                             (64, 3, 128 * SMS, False), (192, 0, 128 * SMS + 1, False), (128, 12, 256 * SMS + 129, False),
                                             (256, 12, 40000, False), (64, 0, 1, True), (256, 4, 63, True), (128, 1, 65, True), (192, 5, 300, True),
                                             (256, 0, 64 * SMS + 1, True), (192, 2, 128 * SMS + 65, True), (64, 6, 256 * SMS + 1, True)])
def test_tensor_core_chain_meets_the_oracle(D, H, lag, S, literal):
    if D == 32:                                          # and widths of other multiples of 32, more than one half of 256
        H = {64: 32, 128: 160, 192: 512, 256: 288 if S % 2 else 448}[H]
    N = 20
    make = inputs.make_weights_literal if literal else inputs.make_weights
    w = make(N, D, H, seed=H + lag, fan_in_ref=32)
    gpu = binding.Cutoff(N, D, H, lag, S, precision=1, seed=3, flags=binding.FLAG_LITERAL if literal else 0)
    gpu.load_weights(w)
    orc = O.CutoffOracle(w, lag, S, seed=3)
    for x in inputs.make_trace(N, lag + 3, seed=S, sigma=0.25):
        gpu.push(x)
        orc.push(x)
    x = gpu.debug_samples(0, S)
    rows = np.unique(np.concatenate([np.linspace(0, S - 1, 150).astype(int), np.arange(max(0, S - 70), S)]))
    ref = orc.samples(rows)
    assert np.max(np.abs(x[rows] - ref) / np.maximum(np.abs(ref), np.abs(ref).mean())) <= 2e-3
    # a sample does not depend on the tile that it is part of
    for first, n in ((0, 1), (S // 3, 65), (S // 2, 64 * SMS + 3)):
        n = min(n, S - first)
        assert np.array_equal(gpu.debug_samples(first, n), x[first:first + n])


# A window of one step is the one in which the tiles of a slot follow each other without a guide step in between: three tiles and more
# for each slot (D = 16: two slots per SM, D = 32: one), all samples against calls that give an SM one tile at most.
@pytest.mark.parametrize("literal", [False, True])
@pytest.mark.parametrize("D,H", [(16, 64), (16, 256), (32, 32), (32, 512)])
def test_tiles_of_a_slot_in_windows_of_one_step(D, H, literal):
    N, S = 20, (256 if D == 16 else 128) * SMS * 3 + 65
    make = inputs.make_weights_literal if literal else inputs.make_weights
    gpu = binding.Cutoff(N, D, H, 0, S, precision=1, seed=7, flags=binding.FLAG_LITERAL if literal else 0)
    gpu.load_weights(make(N, D, H, seed=H, fan_in_ref=32))
    for x in inputs.make_trace(N, 2, seed=D, sigma=0.25):
        gpu.push(x)
    x = gpu.debug_samples(0, S)
    assert np.isfinite(x).all()
    for first in range(0, S, 128 * SMS):
        n = min(128 * SMS, S - first)
        assert np.array_equal(gpu.debug_samples(first, n), x[first:first + n])


# Decisions in passes whose sizes take other kernels than the whole does, chosen after the context was made: whole tiles side by side, then
# one tile per SM and half tiles; the fp32 model with 4, 2 and 1 samples per lane in the emission.
@pytest.mark.parametrize("N,D,H,S,precision,literal", [(20, 16, 128, 40000, 1, False), (20, 16, 128, 40000, 1, True), (20, 32, 64, 40000, 1, False),
                                                       (20, 32, 64, 40000, 1, True), (16, 8, 64, 60000, 0, False), (40, 8, 64, 16000, 0, False)])
def test_decisions_in_passes_of_other_sizes(N, D, H, S, precision, literal):
    make = inputs.make_weights_literal if literal else inputs.make_weights
    gpu = binding.Cutoff(N, D, H, 1, S, precision=precision, seed=7, flags=binding.FLAG_LITERAL if literal else 0)
    gpu.load_weights(make(N, D, H, seed=H, fan_in_ref=32))
    for x in inputs.make_trace(N, 3, seed=D, sigma=0.25):
        gpu.push(x)
    state = gpu.save_state()
    want = np.sort(gpu.debug_samples(0, S).astype(np.float64), axis=1).sum(axis=0)
    for rows in (15000, 8000, 1024):
        gpu.restore_state(state)                                      # the same decision again
        gpu.set_option("pass_rows", rows)
        assert gpu.predict()[0] == binding.OK
        # a warp of the sort adds at most 26 rows (60000 over 296 CTAs of 8) in single precision, warps are added in double: 26 / 2^24
        assert np.max(np.abs(gpu.get_partial_sums() - want)) <= 1.6e-6 * np.abs(want).max()


def test_hidden_layers_keep_their_bits_at_any_scale():
    # the transition's hidden layer times 2^a against output weights times 2^-a: powers of two, so the same samples to the last bit
    N, D, H, lag, S = 20, 16, 128, 2, 2500
    trace = inputs.make_trace(N, lag + 2, seed=4, sigma=0.25)
    out = []
    for a in (0, -40, 40):
        w = inputs.make_weights(N, D, H, seed=9, fan_in_ref=32)
        for k, p in (("W1", a), ("b1", a), ("W2", -a)):
            w[k] = (w[k] * np.float32(2.0 ** p)).astype(np.float32)
        gpu = binding.Cutoff(N, D, H, lag, S, precision=1, seed=3)
        gpu.load_weights(w)
        for x in trace:
            gpu.push(x)
        out.append(gpu.debug_samples(0, S))
    assert np.array_equal(out[1], out[0]) and np.array_equal(out[2], out[0])
