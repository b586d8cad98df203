"""<h|h> of one mode on many knots, to the last bits: how h enters the FP32 pairs of the FP64
path's integrand.

h is rounded to 8 units of 2^-55 of the block's scale, at least 2^-46 of |h| on these
segments, each bin by itself; the bound of all of a walker's bins together is 2^-46 of <h|h>
from that (without the averaging over bins), and the two sides' knots differ by a few
2^-53 (4e-16 each of 10 factors).  1e-14 is their sum.  Cut off at 64 units instead, with half of that in
common, <h|h> was off by up to 3e-14."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f0,days,mass", [(1e-4, 30.0, (5.0, 7.0)), (1e-5, 30.0, (6.0, 7.5)),
                                          (3e-5, 91.3, (5.5, 7.5))])
def test_power_to_the_last_bits(orc, f0, days, mass):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as pkg

    g = W.Grid.spanning(f0, 2e-2, 1.0 / (days * W.DAY_S))
    th = W.draw_walkers(24, 17, mass)
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    d = orc.noise(S, g.df, W.white_noise(g.n_bins, 1))
    t0 = days * W.DAY_S
    _, _, want, _ = orc.loglike(th, t0, [(2, 2)], 1024, g.f0, g.df, d, S)
    like = pkg.LisaLike(modes=[(2, 2)], n_knots=1024, t0=t0, max_batch=24)
    like.set_data(g.f0, g.df, g.n_bins, d, S)
    _, _, hh = like.loglike(th)
    like.close()
    assert np.all(np.abs(hh - want) <= 1e-14 * want)
