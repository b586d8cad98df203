"""The fixed-point dense kernel of the FP64 path where it can go wrong, against the oracle:
grids that end inside a thread's 4 bins, a warp's 128 and a tile's 1024; segments of a few
bins (evaluated in FP64) next to long ones; more segments in a warp's bins than it expands at
a time; mode lists in which modes with the same m are apart, adjacent or alone; tile shapes;
the allocation-free entry point, which converts its data rows as it goes; data that are NaN.

Tolerance: terms are exact to 2^-54 of the block's largest mode, and the scale that bounds a
segment's cubics is loose by at most 2^19 on the shortest segments (8 bins, few knots), so
2^-35 of a term at worst and 1e-13 typically; the two sides' phases differ by rounding
(1e-12 to 1e-9 rad).  1e-9 of the walker's SNR^2 bounds both."""
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


def problem(orc, n_bins, modes, K, B, seed):
    g = W.Grid(1e-4, DF, n_bins)
    th = W.draw_walkers(B, seed, (4.5, 8.0))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    d = orc.template(th[0], W.T0_C1, modes, K, g.f0, g.df, n_bins)
    d = d + orc.noise(S, g.df, W.white_noise(n_bins, seed))
    return g, th, S, d


CASES = [(1, [(2, 2)], 64), (3, [(2, 2)], 16), (125, [(3, 3), (4, 4)], 64), (127, W.MODES6, 64),
         (1021, W.MODES6, 256), (1025, [(3, 2), (2, 1), (2, 2)], 64),
         (4099, [(4, 3), (2, 2), (3, 3), (3, 2)], 300), (20003, W.MODES6, 1024),
         (51581, [(2, 1), (4, 4), (4, 3), (3, 2), (3, 3), (2, 2)], 128)]


@pytest.mark.parametrize("n_bins,modes,K", CASES)
def test_dense_matches_the_oracle(pkg, orc, n_bins, modes, K):
    LL = pkg.lisalike
    g, th, S, d = problem(orc, n_bins, modes, K, 11, n_bins)
    ref, rdh, rhh, dd = orc.loglike(th, W.T0_C1, modes, K, g.f0, g.df, d, S)
    scale = np.maximum(np.maximum(rhh, dd), 1e-300)
    like = pkg.LisaLike(modes=modes, n_knots=K, t0=W.T0_C1, max_batch=11)
    like.set_data(g.f0, g.df, n_bins, d, S)
    for shape in ((8, 8), (4, 8), (8, 1)):
        LL.lisa_like_set_tune(like.h, *shape)
        lnL, dh, hh = like.loglike(th)
        for got, want in ((lnL, ref), (dh, rdh), (hh, rhh)):
            assert np.all(np.abs(got - want) <= 1e-9 * scale), shape
    like.close()


@pytest.mark.parametrize("n_bins,K,bad", [(1021, 256, None), (51581, 1024, None), (1021, 256, 700)])
def test_rows_converted_as_they_are_used(pkg, orc, n_bins, K, bad):
    import torch

    LL = pkg.lisalike
    modes = [(2, 2), (3, 3)]
    g, th, S, d = problem(orc, n_bins, modes, K, 2, 5)
    th[:, 0] = 2e6, 3e6              # bands that reach the top of the grid and hold bin 700
    w = 4.0 * g.df / S
    cols = [w[0], w[1], w[2]]
    for c in range(3):
        cols += [w[c] * d[c].real, w[c] * d[c].imag]
    rows = np.stack(cols, axis=1)
    if bad is not None:
        rows[bad, 4] = np.nan
    cfg = LL.lisa_like_default_config()
    cfg.n_modes, cfg.n_knots, cfg.t0_s = 2, K, W.T0_C1
    for i, (l, m) in enumerate(modes):
        cfg.modes[i][0], cfg.modes[i][1] = l, m
    dd = float(orc.inner(d, d, S, g.df))
    out = torch.empty((3, 2), dtype=torch.float64, device="cuda")
    LL.lisa_like_loglike_noalloc(cfg, g.f0, g.df, n_bins, torch.tensor(rows, device="cuda"), dd,
                                 torch.tensor(th, device="cuda"), 2, out[0], out[1], out[2],
                                 torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    lnL, dh, hh = out.cpu().numpy()
    ref, rdh, rhh, _ = orc.loglike(th, W.T0_C1, modes, K, g.f0, g.df, d, S)
    scale = np.maximum(rhh, dd)
    assert np.all(np.abs(hh - rhh) <= 1e-9 * scale)
    if bad is None:
        assert np.all(np.abs(lnL - ref) <= 1e-9 * scale) and np.all(np.abs(dh - rdh) <= 1e-9 * scale)
    else:
        assert np.all(np.isnan(lnL)) and np.all(np.isnan(dh))
