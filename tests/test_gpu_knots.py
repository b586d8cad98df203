"""Knot values on both sides of the frequency (13 mHz) from which the response's sines are no
longer taken by series, and a grid whose bin numbers are not exact in 64 bits (f / df of 1e12),
against the oracle."""
import numpy as np
import pytest

import workloads as W
from test_gpu_dense import pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmax", [1.2e-2, 1e-1])
def test_knot_values_over_the_band(pkg, orc, fmax):  # noqa: F811
    g = W.Grid.spanning(1e-4, fmax, 1.0 / (30 * W.DAY_S))
    th = W.draw_walkers(6, 12, (4.5, 6.5))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    like = pkg.LisaLike(modes=W.MODES6, n_knots=300, t0=W.T0_C1, max_batch=6)
    like.set_data(g.f0, g.df, g.n_bins, None, orc.psd_aet(g.freqs()))
    band, _, fk, vals = like.stage_knots(th)
    like.close()
    seen = 0
    for b in range(6):
        for mi, (l, m) in enumerate(W.MODES6):
            if not band[b, mi, 0]:
                continue
            seen += 1
            rfk, rvals = orc.knots(th[b], W.T0_C1, l, m, g.f0, g.df, g.n_bins, 300)
            # knots agree to 1e-13 (the band's root), values follow at up to 30 times that and sums of
            # terms of order one at a few 1e-16; the phase reaches 1e5 rad
            assert np.allclose(fk[b, mi], rfk, rtol=1e-12, atol=0)
            for q in range(8):
                scale = np.max(np.abs(rvals[q])) + 1e-300
                assert np.max(np.abs(vals[b, mi, q] - rvals[q])) <= 1e-10 * scale, (b, mi, q)
    assert seen > 20


def test_bin_numbers_that_are_not_exact(pkg, orc):  # noqa: F811
    g = W.Grid(1e-3, 1e-15, 3000)
    th = W.draw_walkers(3, 5, (5.5, 6.0))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    d = orc.template(th[0], W.T0_C1, W.MODES6, 16, g.f0, g.df, g.n_bins)
    ref, rdh, rhh, dd = orc.loglike(th, W.T0_C1, W.MODES6, 16, g.f0, g.df, d, S)
    like = pkg.LisaLike(modes=W.MODES6, n_knots=16, t0=W.T0_C1, max_batch=3)
    like.set_data(g.f0, g.df, g.n_bins, d, S)
    lnL, dh, hh = like.loglike(th)
    like.close()
    assert np.max(rhh) > 0.0
    for got, want in ((lnL, ref), (dh, rdh), (hh, rhh)):
        assert np.all(np.abs(got - want) <= 1e-9 * np.maximum(rhh, dd))
