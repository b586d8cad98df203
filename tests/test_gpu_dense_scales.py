"""<h|h> of the FP64 path where the cubics' third differences are large against their values:
few knots, and grids that begin a few bins above zero frequency.

The fixed-point sums have a unit of at most 2^-41 of the product |A| |T| where a segment
enters a warp's bins, 2^-49 typically, so that <h|h> of one mode, a sum of squares, is right
to about 2^-40 of itself; it does not depend on the phase.  Six modes interfere: there the
two sides' phases (1e-12 rad a mode at these lengths of signal) count.  1e-11 and 1e-10 of
<h|h> itself leave a factor of ten."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

GRIDS = {"month": W.Grid.spanning(1e-5, 2e-2, 1.0 / (30 * W.DAY_S)),
         "week": W.Grid.spanning(1e-4, 2e-2, 1.0 / (7 * W.DAY_S)),
         "coarse": W.Grid(1e-5, 1e-5, 9999)}


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as p

    return p


@pytest.mark.parametrize("modes", [((2, 2),), W.MODES6])
@pytest.mark.parametrize("K", [8, 32, 64, 256])
@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_power_relative_to_itself(pkg, orc, grid, K, modes):
    g = GRIDS[grid]
    th = np.concatenate([W.draw_walkers(12, K, (4.5, 6.5)), W.draw_walkers(12, K + 1, (6.5, 8.0))])
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    th[3, 1] = 1.0   # equal masses: the modes of odd m vanish
    th[15, 6] = 0.0  # face on: only (2, 2) and (3, 2) are seen
    S = orc.psd_aet(g.freqs())
    d = orc.noise(S, g.df, W.white_noise(g.n_bins, 1))
    _, _, want, _ = orc.loglike(th, W.T0_C1, modes, K, g.f0, g.df, d, S)
    like = pkg.LisaLike(modes=modes, n_knots=K, t0=W.T0_C1, max_batch=24)
    like.set_data(g.f0, g.df, g.n_bins, d, S)
    _, _, hh = like.loglike(th)
    like.close()
    assert np.all(np.abs(hh - want) <= (1e-11 if len(modes) == 1 else 1e-10) * want)
