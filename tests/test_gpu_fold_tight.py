"""The fold where the moments of unequal batches would cancel (batches that
scatter by less than a history's mean energy) and where the sum of squares
passes 2^121: both take the two-pass form, against exact rational arithmetic."""
import math
from fractions import Fraction

import numpy as np
import pytest

from tests.gpu_common import need_gpu
from tests.test_gpu_fold_forms import exact, fold

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
N_VOX = 48
CODE = 1 << 24  # 1 g/cm^3: dose and sigma in units of exact()'s scale


def variance_bound(column, n_hist):
    """Relative error of sigma^2.  sigma's constants, reciprocal, square root and
    products: 40 U.  The variance: W + 20 U for its roundings and its sum; the
    rounded mean, off by at most 2 U D, moves it by 2 (2 U D) |sum of the first r
    differences| <= 4 U D sqrt(r acc) and, to second order, W (2 U n_b D)^2; sums
    of 2^53 quanta and more are rounded themselves, 2 U sqrt(sum S^2 / acc)."""
    W, S = len(column), sum(column)
    D = S / n_hist
    n_b = [n_hist // W + (b < n_hist % W) for b in range(W)]
    acc = float(sum((x - n * Fraction(S, n_hist)) ** 2 for x, n in zip(column, n_b)))
    big = 4 * math.sqrt(float(sum(x * x for x in column)) / acc) if max(column) >= 1 << 53 else 0.0
    return (U * (60 + W + 8 * D * math.sqrt((n_hist % W) / acc) + big)
            + 8 * W * (U * max(n_b) * D) ** 2 / acc)


def check(tally, n_hist):
    d, s, _ = fold(tally, np.full(tally.shape[1], CODE, dtype=np.uint32), n_hist)
    for v in range(tally.shape[1]):
        column = [int(x) for x in tally[:, v]]
        dose, var = exact(column, CODE, n_hist)
        assert abs(Fraction(float(d[v])) / dose - 1) < 10 * U
        if var == 0:
            assert s[v] == 0.0
        else:
            assert abs(float(Fraction(float(s[v])) ** 2 / var) - 1) < variance_bound(column, n_hist)


@pytest.mark.parametrize("W", [8, 16, 32, 64])
@pytest.mark.parametrize("extra", [1, 5, -1])
@pytest.mark.parametrize("per_batch,scatter", [(100, 1e-2), (100, 1e-6), (100, 0.0), (10 ** 4, 1e-4), (4000, 1.0),
                                               (3, 0.1), (1, 1e-3)])
def test_tight_unequal_batches(W, extra, per_batch, scatter):
    need_gpu()
    rng = np.random.default_rng([W, extra + 1, per_batch])
    n_hist = W * per_batch + extra
    tally = np.zeros((W, N_VOX), dtype=np.uint64)
    for v in range(N_VOX):
        D = round(2.0 ** rng.uniform(20, 34))  # a history's mean energy in quanta, 1 MeV = 2^26
        for b in range(W):
            n = n_hist // W + (b < n_hist % W)
            tally[b, v] = max(0, n * D + round(scatter * math.sqrt(n) * D * rng.standard_normal()))
    check(tally, n_hist)


@pytest.mark.parametrize("W", [8, 16, 32, 64])
@pytest.mark.parametrize("extra", [0, 1, -1])
def test_sums_of_squares_beyond_128_bits(W, extra):
    need_gpu()
    rng = np.random.default_rng([W, extra + 1])
    tally = rng.integers(0, 1 << 50, (W, N_VOX), dtype=np.uint64)
    for v in range(N_VOX):
        if v % 2 and W <= 32:  # every batch large
            tally[:, v] = (rng.uniform(0.5, 0.9, W) * 2.0 ** 63 / W).astype(np.uint64) * np.uint64(2)
        else:  # two batches hold nearly all
            tally[rng.choice(W, 2, replace=False), v] = rng.integers(1 << 61, 1 << 62, 2, dtype=np.uint64)
    for v in range(N_VOX):
        column = [int(x) for x in tally[:, v]]
        assert sum(column) < 1 << 64 and sum(x * x for x in column) >= 1 << 121
    check(tally, W * 4000 + extra)
