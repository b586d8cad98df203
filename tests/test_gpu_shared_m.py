"""Modes of equal m are evaluated together (knots and relative binning): orders in which they
are apart, alone or in reverse, against the oracle's relative binning, which takes one mode
after the other."""
import numpy as np
import pytest

from oracle import oracle_rb as R
from test_gpu_rb import W, c1_setup, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("modes", [
    [(3, 2)],
    [(3, 2), (2, 2)],
    [(4, 3), (2, 2), (2, 1), (3, 2), (3, 3)],
    [(2, 2), (3, 3), (4, 4), (2, 1), (3, 2), (4, 3)],
])
@pytest.mark.parametrize("n_rb", [8, 100])
def test_relative_binning_of_modes_in_any_order(pkg, orc, modes, n_rb):  # noqa: F811
    g, S, th, d, dd = c1_setup(orc)
    like = pkg.LisaLike(modes=modes, n_knots=64, t0=W.T0_C1, max_batch=8)
    like.set_data(g.f0, g.df, g.n_bins, d, S)
    like.set_fiducial(th, n_rb)
    e = R.edges(th, W.T0_C1, modes, g, n_rb)
    assert np.array_equal(like.rb_edges(), e)
    summ = R.summary(th, W.T0_C1, modes, g, e, d, S)
    X = th * (1 + 1e-4 * np.random.default_rng(7).standard_normal((6, 11)))
    X[0] = th
    lnL, dh, hh = like.loglike_rb(X)
    like.close()
    for b in range(6):
        ref = R.loglike(X[b], th, W.T0_C1, modes, g, e, summ, dd)
        # both sides in 64 bits: phases of 1e5 rad are rounded at 1e-11 rad on either side, and
        # sums of either sign are below hh + dd, so 1e-9 of that holds with a factor of ten
        for got, want in zip((lnL[b], dh[b], hh[b]), ref):
            assert abs(got - want) <= 1e-9 * (abs(hh[b]) + dd)
