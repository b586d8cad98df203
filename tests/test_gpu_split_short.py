"""Split precision on segments of a few bins, of one bin and of none: knots that outnumber the
bins of a band, where a thread's chunk holds several segments and most have no quartics.

Tolerance: the split path's bound against the FP64 path, 1e-6 of SNR^2."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("modes", [((2, 2),), W.MODES6])
@pytest.mark.parametrize("K", [512, 1024, 4096])
def test_short_segments(orc, K, modes):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as pkg

    LL = pkg.lisalike
    g = W.Grid.spanning(1e-4, 5e-3, 1.0 / (7 * W.DAY_S))
    th = W.draw_walkers(21, K, (6.0, 8.0))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    d = orc.noise(S, g.df, W.white_noise(g.n_bins, 1))
    out = {}
    for prec in (pkg.LISA_PREC_FP64, pkg.LISA_PREC_SPLIT):
        like = pkg.LisaLike(modes=modes, n_knots=K, t0=7 * W.DAY_S, max_batch=21, precision=prec)
        like.set_data(g.f0, g.df, g.n_bins, d, S)
        for shape in ((8, 8), (4, 8), (8, 1)) + (((16, 8),) if prec == pkg.LISA_PREC_SPLIT else ()):
            LL.lisa_like_set_tune(like.h, *shape)
            out[prec, shape] = np.stack(like.loglike(th))
        dd = like.data_inner()
        like.close()
    ref = out[pkg.LISA_PREC_FP64, (8, 8)]
    for got in out.values():
        assert np.all(np.abs(got[:2] - ref[:2]) <= 1e-6 * np.maximum(ref[2], dd))
        assert np.all(np.abs(got[2] - ref[2]) <= 1e-6 * ref[2])
