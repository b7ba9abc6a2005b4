"""The guided search of a spectrum's CDF finds the bin the whole search does:
the first whose end reaches the quantile, for one bin, the most bins, bins of no
weight at either end and between, and bins far narrower than a guide cell."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import make_ctx

pytestmark = pytest.mark.gpu

_R = np.random.default_rng(4)
WEIGHTS = {
    "one": np.array([3.0]),
    "two": np.array([1.0, 1e-6]),
    "flat14": np.full(14, 1.0 / 14),
    "gaps": np.array([0.0, 0.0, 1.0, 0.0, 0.5, 0.0, 0.0, 2.0, 0.0]),
    "6mv": W.synthetic_6mv_spectrum()[1],
    "1024": _R.random(1024),
    "spike": np.where(np.arange(1024) == 700, 1.0, 1e-7),
    "sparse": np.where(_R.random(1023) < 0.9, 0.0, _R.random(1023)),
}


@pytest.mark.parametrize("name", sorted(WEIGHTS))
def test_bins_equal_the_whole_search(name):
    w, n, seed = WEIGHTS[name], 200_003, 77
    edges = np.linspace(0.5, 12.0, len(w) + 1)
    src = W.Source(W.PHOTON, W.BEAM_SQUARE, spectrum_edges=edges, spectrum_weights=w)
    ctx = make_ctx()
    e = ctx.debug_sample(5, 0.0, n, seed, src=src)
    ctr = np.zeros((n, 4), dtype=np.uint32)
    ctr[:, 2] = 0x5EED
    ctr[:, 3] = np.arange(n)
    word = ctx.debug_philox(ctr, [seed, 0], use_curand=True)[:, 2]
    ctx.close()
    z = (((word >> 8).astype(np.float64) + 1.0) * 2.0 ** -24).astype(np.float32)
    cdf = (np.cumsum(w) / np.cumsum(w)[-1]).astype(np.float32)
    cdf[-1] = 1.0
    k = np.minimum(np.searchsorted(cdf, z, side="left"), len(w) - 1)  # first bin whose end reaches z
    ef = edges.astype(np.float32)
    assert np.all(w[k] > 0)
    assert np.all(e >= ef[k]) and np.all(e <= ef[k + 1])
