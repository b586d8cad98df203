"""The split-precision dense kernel where it can go wrong, against the oracle: grids that end
inside a thread's chunk, a warp's and a tile; bands that end inside them; segments shorter than
a chunk, longer than a warp's bins and longer than 65536 bins; few knots, where the modes of an
m are evaluated one by one instead of as one quartic; mode lists in which modes with the
same m are apart, adjacent or alone; every tile shape.

Tolerance: amplitude, transfer, phasor and their products are rounded to FP32 (about ten
roundings of 2^-24, 6e-7 if all had one sign), so 1e-6 of the walker's SNR^2."""
import numpy as np
import pytest

import workloads as W
from test_gpu_dense import pkg, problem  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins,modes,K", [
    (1, [(2, 2)], 64), (7, [(3, 2)], 16), (1021, W.MODES6, 64), (1025, [(3, 2), (2, 1), (2, 2)], 300),
    (4099, [(4, 3), (2, 2), (3, 3), (3, 2)], 16), (20003, W.MODES6, 1024),
    (51581, [(2, 1), (4, 4), (4, 3), (3, 2), (3, 3), (2, 2)], 128), (300007, [(2, 2), (3, 3)], 24),
    (300007, W.MODES6, 512)])
def test_split_matches_the_oracle(pkg, orc, n_bins, modes, K):  # noqa: F811
    LL = pkg.lisalike
    g, th, S, d = problem(orc, n_bins, modes, K, 11, n_bins)
    ref, rdh, rhh, dd = orc.loglike(th, W.T0_C1, modes, K, g.f0, g.df, d, S)
    scale = np.maximum(np.maximum(rhh, dd), 1.0)
    like = pkg.LisaLike(modes=modes, n_knots=K, t0=W.T0_C1, max_batch=11, precision=pkg.LISA_PREC_SPLIT)
    like.set_data(g.f0, g.df, n_bins, d, S)
    for shape in ((8, 8), (4, 8), (16, 8), (8, 1)):
        LL.lisa_like_set_tune(like.h, *shape)
        lnL, dh, hh = like.loglike(th)
        for got, want in ((lnL, ref), (dh, rdh), (hh, rhh)):
            assert np.all(np.abs(got - want) <= 1e-6 * scale), shape
    like.close()
