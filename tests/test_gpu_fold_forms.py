"""The FP64 fold against exact rational arithmetic: dose and sigma of synthetic
batch tallies, for every batch count, with equal and unequal batches, from
single deposits to sums beyond the 128-bit form, and the integer outputs."""
import ctypes as C
import math
from fractions import Fraction

import numpy as np
import pytest

import paper_1101_1245_gb300 as g
from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu

INV_VOL = 1.0 / 0.3 ** 3
# gm::launch_fold(tally, vox, nvox, W, n_hist, inv_vol, dose, sigma, dmax_bits, dep_sum, n_sm, stream)
SYMBOL = "_ZN2gm11launch_foldEPKyPKjmimdPdS4_PyS5_iP11CUstream_st"
UNIT = Fraction(1, 2 ** 26) * Fraction(1.602176634e-10) * Fraction(INV_VOL)


def fold(tally, codes, n_hist):
    import torch
    W, nvox = tally.shape
    t = torch.from_numpy(tally.view(np.int64)).cuda()
    v = torch.from_numpy((codes << 4).astype(np.uint32).view(np.int32)).cuda()
    d = torch.empty(nvox, dtype=torch.float64, device="cuda")
    s = torch.empty_like(d)
    red = torch.zeros(2, dtype=torch.int64, device="cuda")
    f = getattr(g.lib(), SYMBOL)
    f.restype = C.c_int
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_uint64, C.c_int, C.c_uint64, C.c_double, C.c_void_p, C.c_void_p,
                  C.c_void_p, C.c_void_p, C.c_int, C.c_void_p]
    torch.cuda.synchronize()
    assert f(t.data_ptr(), v.data_ptr(), nvox, W, n_hist, INV_VOL, d.data_ptr(), s.data_ptr(), red.data_ptr(),
             red.data_ptr() + 8, 152, None) == 0
    torch.cuda.synchronize()
    return d.cpu().numpy(), s.cpu().numpy(), red.cpu().numpy()


def exact(column, code, n_hist):
    """(dose, sigma^2) of a voxel as fractions."""
    W, S = len(column), sum(column)
    D = Fraction(S, n_hist)
    acc = sum((x - (n_hist // W + (1 if b < n_hist % W else 0)) * D) ** 2 for b, x in enumerate(column))
    scale = UNIT * 2 ** 24 / code
    return D * scale, acc * Fraction(W, (W - 1) * n_hist ** 2) * scale * scale


def tallies(W, size, rng):
    """Batch sums about `size`: sparse (a few deposits), Poisson-like and tight (0.1%) columns, and zeros."""
    n = 96
    t = np.zeros((W, n), dtype=np.uint64)
    for v in range(n):
        kind = v % 4
        if kind == 0:  # one to three deposits
            for b in rng.integers(0, W, 1 + v % 3):
                t[b, v] = int(rng.integers(1, size + 1))
        elif kind == 1:
            t[:, v] = rng.integers(0, size + 1, W, dtype=np.uint64)
        elif kind == 2:
            t[:, v] = (size * (1.0 + 1e-3 * rng.standard_normal(W))).astype(np.uint64)
    return t


@pytest.mark.parametrize("W", [8, 16, 32, 64])
@pytest.mark.parametrize("extra", [0, 1, 5, -1])
@pytest.mark.parametrize("size", [3, 2 ** 20, 2 ** 34, 2 ** 45, 2 ** 57])
def test_fold_equals_exact_arithmetic(W, extra, size):
    need_gpu()
    rng = np.random.default_rng(W * 1000 + extra + size % 97)
    tally = tallies(W, size, rng)
    n_hist = W * 4000 + extra
    codes = rng.integers(1, 1 << 28, tally.shape[1]).astype(np.uint32)
    codes[:6] = (1, 2, 3, (1 << 24) + 1, (1 << 28) - 1, 1 << 27)
    d, s, red = fold(tally, codes, n_hist)
    assert int(red[1]) % 2 ** 64 == int(tally.sum())  # as unsigned
    assert red[0] == d.view(np.int64).max()
    for v in range(tally.shape[1]):
        want, var = exact([int(x) for x in tally[:, v]], int(codes[v]), n_hist)
        if want == 0:
            assert d[v] == 0.0 and s[v] == 0.0
            continue
        # dose: the sum, two constants of three or four operations, a
        # reciprocal and two products, each within an ulp: under 10 half-ulps
        assert abs(Fraction(float(d[v])) / want - 1) < 10 * 2.0 ** -53
        # sigma: the same, a square root, and (unequal batches) the variance's
        # last three operations, whose terms are no larger than it
        if var:
            assert abs(float(Fraction(float(s[v])) ** 2 / var) - 1) < 2 * 20 * 2.0 ** -53
        else:
            assert s[v] <= 1e-12 * d[v]


def test_fewer_histories_than_batches():
    need_gpu()
    W, n_hist = 16, 5
    tally = np.zeros((W, 4), dtype=np.uint64)
    tally[:5, 0] = 7, 0, 3, 1, 9
    tally[0, 1] = 1
    tally[4, 2] = 2 ** 40
    d, s, _ = fold(tally, np.full(4, 1 << 24, dtype=np.uint32), n_hist)
    for v in range(3):
        want, var = exact([int(x) for x in tally[:, v]], 1 << 24, n_hist)
        assert abs(Fraction(float(d[v])) / want - 1) < 10 * 2.0 ** -53
        assert math.isclose(float(s[v]), math.sqrt(var), rel_tol=20 * 2.0 ** -53)
    assert d[3] == 0.0 and s[3] == 0.0
