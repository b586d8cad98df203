"""set_data with graphs on: the next call of the same batch size sees the new data and grid,
not the captured ones.  Same bits as a handle that has only seen the new data."""
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


@pytest.mark.parametrize("precision", ["LISA_PREC_FP64", "LISA_PREC_SPLIT"])
@pytest.mark.parametrize("n_bins", [3001, 4003])  # the same grid with other data; another grid
def test_new_data_after_a_capture(pkg, orc, precision, n_bins):
    import torch

    LL = pkg.lisalike
    prec = getattr(pkg, precision)
    th = W.draw_walkers(5, 3, (5.5, 7.0))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]

    def handle():
        return pkg.LisaLike(modes=W.MODES6, n_knots=64, t0=W.T0_C1, max_batch=5, precision=prec)

    def data(n, seed):
        g = W.Grid(1e-4, 1.0 / (30 * W.DAY_S), n)
        S = orc.psd_aet(g.freqs())
        return g.f0, g.df, n, orc.noise(S, g.df, W.white_noise(n, seed)), S

    a, b = handle(), handle()
    a.set_data(*data(3001, 1))
    LL.lisa_like_set_graphs(a.h, True)
    a.loglike(th)                                   # capture with host buffers
    a.set_data(*data(n_bins, 2))
    b.set_data(*data(n_bins, 2))
    want = b.loglike(th)
    for _ in range(2):
        assert all(np.array_equal(x, y) for x, y in zip(a.loglike(th), want))
    dp = torch.tensor(th, device="cuda")
    out = torch.empty((3, 5), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    LL.lisa_like_loglike_device(a.h, dp, 5, out[0], out[1], out[2], st)   # capture with these
    a.set_data(*data(3001, 1))
    b.set_data(*data(3001, 1))
    LL.lisa_like_loglike_device(a.h, dp, 5, out[0], out[1], out[2], st)
    torch.cuda.synchronize()
    assert all(np.array_equal(x, y) for x, y in zip(out.cpu().numpy(), b.loglike(th)))
    a.close()
    b.close()
