"""A band that begins one bin below its first knot: the band rule takes a bin up to 1e-9 bins
below the starting frequency, the first segment the first bin at or above it.  In the FP64
dense kernel the thread that owns such a bin, where its index is 3 modulo 4, begins four bins
before the segment does; every index modulo 4 is tried.

The PSD is the template's own power in A and E, so that every bin of the band weighs the
same: one wrong bin of about 1900 moves <h|h> by 5e-4.  Tolerance: the two sides differ by the
rounding of the phases (1e-12 to 1e-9 rad) and amplitudes (1e-13); 1e-9 of SNR^2 bounds both."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

DF = 1.0 / (30 * W.DAY_S)


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as p

    return p


def at_bin(orc, th, g, j):
    """th with the t_ref that puts the (2,2) mode's start half of 1e-9 bins above bin j."""
    want = g.f0 + j * g.df + 5e-10 * g.df
    lo, hi = -20 * W.DAY_S, 60 * W.DAY_S  # the start falls as t_ref grows
    th = th.copy()
    for _ in range(200):
        th[10] = 0.5 * (lo + hi)
        r = orc.band(th, W.T0_C1, 2, 2, g.f0, g.df, g.n_bins)
        if r is None or r[0] > want:
            lo = th[10]
        else:
            hi = th[10]
    return th


@pytest.mark.parametrize("residue", [0, 1, 2, 3])
def test_bin_below_the_first_knot(pkg, orc, residue):
    LL = pkg.lisalike
    g = W.Grid(1e-4, DF, 2003)
    base = np.array([2e6, 0.4, 0.2, -0.3, 15.0, 1.0, 1.1, 0.7, 0.4, 0.9, 0.0])
    first = orc.band(base, W.T0_C1, 2, 2, g.f0, g.df, g.n_bins)[2]
    j = first + 40 + (residue - first - 40) % 4
    th = at_bin(orc, base, g, j)
    h = orc.template(th, W.T0_C1, [(2, 2)], 64, g.f0, g.df, g.n_bins)
    S = np.abs(h) ** 2
    S[2] = S[0]  # T is a difference of nearly equal terms here: eight digits of it are rounding
    S[:, :j] = S[:, j:j + 1]
    d = 1.5 * h
    ref, rdh, rhh, dd = orc.loglike(th[None], W.T0_C1, [(2, 2)], 64, g.f0, g.df, d, S)
    like = pkg.LisaLike(modes=[(2, 2)], n_knots=64, t0=W.T0_C1, max_batch=8)
    like.set_data(g.f0, g.df, g.n_bins, d, S)
    band, _, fk, _ = like.stage_knots(th)
    assert band[0, 0, 1] == j and j % 4 == residue
    assert fk[0, 0, 0] > g.f0 + j * g.df  # the bin is below the first knot
    assert np.sum(g.freqs() < fk[0, 0, 1]) - j > 8  # a segment that the expansions take
    for shape in ((8, 8), (4, 8), (8, 1)):
        LL.lisa_like_set_tune(like.h, *shape)
        lnL, dh, hh = like.loglike(np.repeat(th[None], 3, axis=0))
        for got, want in ((lnL, ref), (dh, rdh), (hh, rhh)):
            assert np.all(np.abs(got - want[0]) <= 1e-9 * max(rhh[0], dd)), shape
    like.close()
