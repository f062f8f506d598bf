"""The row sorts of the decision and of the allocation-free entry point against numpy's sort, at the row lengths where the
kernels change (keys per thread, warps per row, network or buckets) and on rows their bucket map cannot spread.

A sum of R sorted values is formed by at most 64 (static call: by contract; decisions: R / warps in the grid) fp32 additions
per warp and up to 24 more per CTA, then in double: relative error at most (64 + 24) * 2^-24 = 5e-6 of the sum of magnitudes.
"""
import numpy as np
import pytest

from paper_1803_04209_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu

REL = 5e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "these tests need a GPU"
    build.build()
    return binding.load_library()


def _rows(kind, rows, n, rng):
    x = (0.5 + 0.1 * rng.standard_normal(n) + 0.05 * rng.standard_normal((rows, n))).astype(np.float32)
    if kind == "ties":
        x = (np.round(x * 32) / 32).astype(np.float32)
    elif kind == "equal rows":
        x[::3] = 0.25
    elif kind == "far clusters":
        x = (x * 1e-3 + np.where(np.arange(n) % 2, 1000.0, 0.0)).astype(np.float32)
    elif kind == "heavy tails":
        x = (x / (rng.random((rows, n)) + 1e-4) * np.where(rng.random((rows, n)) < 0.5, -1, 1)).astype(np.float32)
    elif kind == "changing scale":
        x *= (10.0 ** rng.integers(-6, 6, size=(rows, 1))).astype(np.float32)
    elif kind == "infinities":
        x[rng.random((rows, n)) < 0.02] = np.inf
    return x


def _check(got, x):
    s = np.sort(x, axis=1).astype(np.float64)
    want, size = s.sum(axis=0), np.abs(s).sum(axis=0)
    finite = np.isfinite(want)
    assert np.array_equal(finite, np.isfinite(got))
    assert np.all(np.abs(got[finite] - want[finite]) <= REL * size[finite])


@pytest.mark.parametrize("n,rows,pad", [(128, 40, 0), (129, 40, 3), (129, 8192, 3), (256, 8200, 0), (257, 1, 0), (257, 500, 1), (384, 3, 0),
                                        (385, 300, 0), (512, 300, 5), (513, 300, 3), (640, 300, 0), (641, 300, 0), (768, 300, 0),
                                        (769, 300, 7), (896, 300, 0), (897, 300, 2), (1023, 5000, 1), (1024, 5000, 0)])
def test_static_row_sums_at_the_edges_of_the_kernels(n, rows, pad):
    import torch
    x = _rows("plain", rows, n + pad, np.random.default_rng(n + rows))
    sums = torch.empty(n, dtype=torch.float64, device="cuda")
    binding.sorted_row_sums_static(torch.from_numpy(x).cuda(), sums, n=n)
    _check(sums.cpu().numpy(), x[:, :n])


@pytest.mark.parametrize("kind", ["ties", "equal rows", "far clusters", "heavy tails", "changing scale", "infinities"])
@pytest.mark.parametrize("n", [300, 700, 1024])
def test_static_row_sums_of_rows_the_buckets_do_not_spread(kind, n):
    import torch
    x = _rows(kind, 5000, n, np.random.default_rng(n))
    sums = torch.empty(n, dtype=torch.float64, device="cuda")
    binding.sorted_row_sums_static(torch.from_numpy(x).cuda(), sums)
    _check(sums.cpu().numpy(), x)


def test_static_row_sums_from_an_unaligned_base():
    import torch
    flat = _rows("plain", 1, 300 * 704 + 1, np.random.default_rng(5)).reshape(-1)
    x = torch.from_numpy(flat).cuda()[1:].view(300, 704)
    sums = torch.empty(700, dtype=torch.float64, device="cuda")
    binding.sorted_row_sums_static(x, sums, n=700)
    _check(sums.cpu().numpy(), flat[1:].reshape(300, 704)[:, :700])


@pytest.mark.parametrize("N,S,std", [(128, 300, False), (129, 8192, False), (200, 300, True), (257, 100, False), (300, 5000, True), (512, 3000, False),
                                     (641, 3000, False), (897, 1000, True), (1024, 4000, False), (1025, 700, False), (1536, 900, True),
                                     (1537, 700, False), (2048, 900, False), (2049, 900, True), (2560, 700, False), (2561, 700, False),
                                     (3072, 300, True), (3584, 700, False), (3585, 700, False), (4096, 1300, True), (4096, 1, False)])
def test_decision_sums_equal_the_sorted_draws(N, S, std):
    wl = inputs.WORKLOADS["n1024"]
    ctx = binding.Cutoff(N, 4, 32, 1, S, precision=0, seed=N)
    ctx.load_weights(inputs.make_weights(N, 4, 32, seed=N, fan_in_ref=32))
    if std:
        ctx.set_option("order_stat_std", 1)
    for x in inputs.make_trace(N, 2, 7, **wl.trace):
        ctx.push(x)
    draws = ctx.debug_samples(0, S)
    ctx.predict()
    _check(ctx.get_partial_sums(), draws)
    if std:
        scale = float(ctx.get_stats()[0][-1]) / float(np.sort(draws, axis=1)[:, -1].astype(np.float64).mean())
        want = np.sort(draws, axis=1).astype(np.float64).std(axis=0) * scale
        # a difference of two sums of squares: the sums' 5e-6, over twice the deviation
        bound = 1e-5 + REL * (np.square(draws.astype(np.float64)).max() * scale * scale) / (2 * want)
        assert np.all(np.abs(ctx.get_order_stat_std() - want) <= bound)
    ctx.close()


@pytest.mark.parametrize("N,S", [(300, 700), (1024, 5000), (2175, 1500), (4096, 1300)])
def test_decision_sums_of_tied_and_clustered_draws(N, S):
    """A model without noise whose workers take a handful of values, so that most keys of a row are equal or far from
    the others: the bucket map cannot spread them."""
    w = inputs.make_weights(N, 4, 32, seed=1, fan_in_ref=32)
    w["W4"][:] = 0.0
    w["b4"][:N] = np.random.default_rng(N).choice([0.25, 0.5, 0.50001, 300.0], size=N)
    w["b4"][N:] = -200.0
    ctx = binding.Cutoff(N, 4, 32, 1, S, precision=0, seed=N)
    ctx.load_weights(w)
    for x in inputs.make_trace(N, 2, 7, sigma=0.3):
        ctx.push(x)
    draws = ctx.debug_samples(0, S)
    ctx.predict()
    _check(ctx.get_partial_sums(), draws)
    ctx.close()


def _one_value_decision(N, S, v):
    w = inputs.make_weights(N, 4, 32, seed=1, fan_in_ref=32)
    w["W4"][:] = 0.0
    w["b4"][:N] = v
    w["b4"][N:] = -400.0                                  # every draw is v exactly
    ctx = binding.Cutoff(N, 4, 32, 1, S, precision=0, seed=N)
    ctx.load_weights(w)
    for x in inputs.make_trace(N, 2, 7, sigma=0.3):
        ctx.push(x)
    ctx.predict()
    sums = ctx.get_partial_sums()
    ctx.close()
    return sums


# The warps of a CTA are added in double and rounded to single once: half a unit in the last place of the CTA's sum, 2^-24 relative.
@pytest.mark.parametrize("N,S", [(130, 65536), (300, 65536), (700, 65536), (1024, 65536)])
def test_the_warps_of_a_cta_are_added_in_double(N, S):
    for v in (1 + 2.0 ** -18, 1 + 3 * 2.0 ** -18, 1 + 5 * 2.0 ** -17, 1.5 + 2.0 ** -18):
        sums = _one_value_decision(N, S, np.float32(v))
        assert np.all(np.abs(sums - S * v) <= 2.0 ** -24 * S * v), v


@pytest.mark.parametrize("n", [130, 300, 700, 1024])
def test_the_warps_of_a_cta_of_the_static_call_are_added_in_double(n):
    import torch
    sums = torch.empty(n, dtype=torch.float64, device="cuda")
    for v in (1 + 2.0 ** -18, 1 + 3 * 2.0 ** -18, 1 + 5 * 2.0 ** -17):
        x = torch.full((131072 + 70000, n + 1), v, dtype=torch.float32, device="cuda")
        for rows, tolerance in ((65536, 2.0 ** -24), (x.shape[0], REL)):           # one block of rows; two, the first with chains beyond 32
            for y in (x[:rows, :n], x.view(-1)[: rows * n].view(rows, n)):
                binding.sorted_row_sums_static(y, sums, n=n)
                assert np.all(np.abs(sums.cpu().numpy() - rows * v) <= tolerance * rows * v), (rows, v)


# A thread of a wide decision adds 4 rows in single precision, then those to its totals, whose rounding is carried on: 4 copies of a
# value of 21 bits add up without rounding, so all that is lost is the one rounding of a CTA's result.
@pytest.mark.parametrize("N", [1025, 1537, 2049, 2561, 3073, 4096])
def test_wide_decisions_keep_their_single_precision_sums_short(N):
    for v in (1 + 2.0 ** -19, 1 + 3 * 2.0 ** -20):
        sums = _one_value_decision(N, 32768, np.float32(v))
        assert np.all(np.abs(sums - 32768 * v) <= 2.0 ** -24 * 32768 * v), v


# rows per thread around multiples of the 4 that are added in registers, in one pass and in several; squares too
@pytest.mark.parametrize("N,S,pass_rows", [(1100, 888 * 3, 0), (1100, 888 * 4, 0), (1100, 888 * 8, 0), (1700, 740 * 9 - 1, 0), (4096, 592 * 16, 0), (4096, 592 * 16 + 1, 0),
                                           (2200, 20000, 0), (3000, 30000, 10000), (3500, 9000, 1024)])
def test_wide_decisions_around_the_length_of_a_run(N, S, pass_rows):
    got = []
    for std in (0, 1):
        ctx = binding.Cutoff(N, 4, 32, 1, S, precision=0, seed=N)
        ctx.load_weights(inputs.make_weights(N, 4, 32, seed=N, fan_in_ref=32))
        ctx.set_option("order_stat_std", std)
        if pass_rows:
            ctx.set_option("pass_rows", pass_rows)
        for x in inputs.make_trace(N, 2, 7, sigma=0.3):
            ctx.push(x)
        want, size, squares = np.zeros(N), np.zeros(N), np.zeros(N)
        for k in range(0, S if std else 0, 4096):
            draws = np.sort(ctx.debug_samples(k, min(4096, S - k)), axis=1).astype(np.float64)
            want, size, squares = want + draws.sum(axis=0), size + np.abs(draws).sum(axis=0), squares + (draws * draws).sum(axis=0)
        ctx.predict()
        got.append(ctx.get_partial_sums())
    assert np.array_equal(got[0], got[1])                 # the sums do not depend on the squares
    assert np.all(np.abs(got[1] - want) <= REL * size)
    scale = float(ctx.get_stats()[0][-1]) * S / want[-1]
    sd = np.sqrt(squares / S - (want / S) ** 2) * scale
    assert np.all(np.abs(ctx.get_order_stat_std() - sd) <= 1e-5 + REL * squares / S * scale * scale / (2 * sd))
@pytest.mark.parametrize("n,rows", [(160, 9000), (256, 9000), (300, 6000), (700, 6000), (1000, 6000)])
def test_rows_that_change_between_spread_and_not(n, rows):
    # a warp's rows take turns: ones the map spreads, ones it does not, and neighbours of another scale
    import torch
    rng = np.random.default_rng(n)
    x = _rows("plain", rows, n, rng)
    turn = rng.integers(0, 4, rows)
    x[turn == 0] = np.float32(0.75)
    x[turn == 1] *= np.float32(1e3)
    x[rows // 2: rows // 2 + rows // 4] = np.float32(0.5)
    sums = torch.empty(n, dtype=torch.float64, device="cuda")
    binding.sorted_row_sums_static(torch.from_numpy(x).cuda(), sums)
    _check(sums.cpu().numpy(), x)


# Row by row and bit for bit, at the edges of the keys per thread: a warp (CTA) sorts rows of all kinds in turn, so that rows meet the
# bucket map of another kind and scale.  129 to 256 keys take the buckets from 8192 rows on.
@pytest.mark.parametrize("n,rows", [(128, 90), (129, 8192), (200, 8191), (256, 8200)] +
                         [(n, 90) for e in range(8, 32, 4) for n in (32 * e, 32 * e + 1)] + [(1023, 90), (1024, 90)] +
                         [(n, 90) for e in range(8, 32, 4) for n in (128 * e + 1, 128 * e + 128 * 4)] + [(2175, 90), (4095, 90)])
def test_sorted_rows_bit_for_bit(n, rows):
    rng = np.random.default_rng(n)
    kinds = [_rows(k, rows, n, rng) for k in ("plain", "ties", "equal rows", "far clusters", "heavy tails", "changing scale", "infinities")]
    kinds.append(np.where(rng.random((rows, n)) < 0.5, 0.0, -0.0).astype(np.float32))
    kinds.append(np.sort(kinds[0], axis=1)[:, ::-1])
    x = np.stack(kinds)[rng.integers(0, len(kinds), rows), np.arange(rows)]
    ctx = binding.Cutoff(16, 4, 32, 1, 64)
    got, want = ctx.debug_sort_values(x), np.sort(x, axis=1)
    nonzero = want != 0
    assert np.array_equal(got, want)
    assert np.array_equal(got.view(np.uint32)[nonzero], want.view(np.uint32)[nonzero])
    zeros = ~nonzero
    assert np.array_equal(np.signbit(got).sum(axis=1), np.signbit(x).sum(axis=1))           # -0 before +0, none lost
    for r in np.flatnonzero(zeros.any(axis=1)):
        sign = np.signbit(got[r][zeros[r]])
        assert np.all(sign[:-1] >= sign[1:])
