"""The chunked spline solve against the oracle's serial one on the device's own knot values.

Sizes: the smallest systems, one row either side of the 34 knots from which a sweep no
longer starts at the first row, chunk edges, and the sizes from which a system is dealt to
two, four and eight blocks (few systems, or rows that no longer fit in shared memory).

Tolerance: the solves differ by the rounding of sums of the same terms (a few 1e-16 of the
slopes' differences) and by the run-in (0.36^32 < 1e-14 of a neighbour's value); the
interpolant takes h^2 M / 8 of that, so 1e-12 of the series' scale leaves a factor of 100."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as p

    return p


@pytest.mark.parametrize("K,B", [(4, 1), (5, 60), (33, 1), (34, 60), (35, 1), (36, 20), (66, 60),
                                 (257, 1), (509, 10), (1023, 60), (1025, 20), (2400, 60), (4096, 60)])
def test_chunked_solve_matches_the_serial_one(pkg, orc, K, B):
    g = W.Grid.spanning(1e-4, 2e-2, 1.0 / (30 * W.DAY_S))
    th = W.draw_walkers(B, 31)
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    like = pkg.LisaLike(modes=W.MODES6, n_knots=K, t0=W.T0_C1, max_batch=B)
    like.set_data(g.f0, g.df, g.n_bins, None, orc.psd_aet(g.freqs()))
    band, _, fk, vals = like.stage_knots(th)
    coef = like.stage_coeffs(th)
    like.close()
    seen = 0
    for b, mi in ((0, 0), (0, 5), (B // 2, 3), (B - 1, 1)):
        if not band[b, mi, 0]:
            continue
        seen += 1
        h = np.diff(fk[b, mi])
        for q in range(8):
            ref = orc.spline(fk[b, mi], vals[b, mi, q])
            scale = np.max(np.abs(vals[b, mi, q])) + 1e-300
            for frac in (0.0, 0.5, 1.0):
                x = (frac * h)[:, None] ** np.arange(4)[None, :]
                diff = np.sum((coef[b, mi, :, q, :] - ref) * x, axis=1)
                assert np.max(np.abs(diff)) <= 1e-12 * scale, (b, mi, q, frac)
    assert seen


@pytest.mark.parametrize("K", [35, 2400, 4096])
def test_split_records_at_the_same_sizes(pkg, orc, K):
    """The split-precision records of the same splines: ln L within its 1e-6 SNR^2 bound."""
    g = W.Grid.spanning(1e-4, 2e-2, 1.0 / (30 * W.DAY_S))
    th = W.draw_walkers(12, 32)
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    d = orc.template(th[1], W.T0_C1, W.MODES6, 64, g.f0, g.df, g.n_bins)
    out = []
    for prec in (pkg.LISA_PREC_FP64, pkg.LISA_PREC_SPLIT):
        like = pkg.LisaLike(modes=W.MODES6, n_knots=K, t0=W.T0_C1, max_batch=12, precision=prec)
        like.set_data(g.f0, g.df, g.n_bins, d, S)
        out.append(like.loglike(th))
        dd = like.data_inner()
        like.close()
    scale = np.maximum(np.maximum(out[0][2], dd), 1.0)
    assert np.all(np.abs(out[1][0] - out[0][0]) <= 1e-6 * scale)
