"""FP64 handles without their second copy of the data: rows converted as they are used, one
walker per item; and the copy's room, which any other allocation may have.

The two paths evaluate the same fixed-point sums from other origins, each to 2^-45 of a
thread's sum and one rounding in FP64 per sum: 1e-12 of SNR^2."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    import paper_2005_01827_gb300 as p

    return p


def problem(orc, n, B):
    g = W.Grid(1e-4, 0.02 / n, n)
    th = W.draw_walkers(B, n, (5.0, 7.0))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    S = orc.psd_aet(g.freqs())
    return (g.f0, g.df, n, orc.noise(S, g.df, W.white_noise(n, 1)), S), th


def same(a, b, dd):
    return all(np.all(np.abs(x - y) <= 1e-12 * np.maximum(b[2], dd)) for x, y in zip(a, b))


@pytest.mark.parametrize("n", [1021, 51583])
def test_without_the_second_copy(pkg, orc, monkeypatch, n):
    LL = pkg.lisalike
    data, th = problem(orc, n, 11)
    like = pkg.LisaLike(n_knots=64, t0=W.T0_C1, max_batch=11)
    like.set_data(*data)
    want, dd = like.loglike(th), like.data_inner()
    assert LL.lisa_like_get_tune(like.h)[1] == 8
    LL.lisa_like_set_graphs(like.h, True)
    like.loglike(th)
    monkeypatch.setenv("LISA_LIKE_ONE_COPY", "1")
    like.set_data(*data)
    for shape in ((8, 8), (4, 8), (8, 1)):
        LL.lisa_like_set_tune(like.h, *shape)
        assert list(LL.lisa_like_get_tune(like.h))[:2] == [shape[0], 1]
        assert same(like.loglike(th), want, dd)
    assert LL.lisa_like_autotune(like.h, th, 11)[1] == 1
    monkeypatch.delenv("LISA_LIKE_ONE_COPY")
    like.set_data(*data)
    LL.lisa_like_set_tune(like.h, 8, 8)
    assert LL.lisa_like_get_tune(like.h)[1] == 8
    assert all(np.array_equal(x, y) for x, y in zip(like.loglike(th), want))
    like.close()


def test_room_for_others_comes_first(pkg, orc):
    import torch

    LL = pkg.lisalike
    n = 4000003
    data, th = problem(orc, n, 2)
    rows, bins, up = 76 * n, 72 * n, 72 * n  # second copy, data, PSD and d on their way

    def leave(nbytes):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")

    like = pkg.LisaLike(n_knots=64, t0=W.T0_C1, max_batch=2)
    like.set_data(*data)
    want, dd = like.loglike(th), like.data_inner()
    assert LL.lisa_like_get_tune(like.h)[1] == 8
    hog = leave(bins + up // 2)  # enough for new data only with the old second copy's room
    like.set_data(*data)
    assert same(like.loglike(th), want, dd)
    del hog
    torch.cuda.empty_cache()
    like.set_data(*data)
    assert LL.lisa_like_get_tune(like.h)[1] == 8
    hog = leave(16 * MIB)        # not enough at all: refused, and the old data are still in use
    with pytest.raises(pkg.lisalike.LisaError):
        like.set_data(*data)
    assert same(like.loglike(th), want, dd)
    del hog
    torch.cuda.empty_cache()
    like.close()
    hog = leave(bins + up + rows // 2 + 64 * MIB)  # the data fit, the second copy is not worth it
    like = pkg.LisaLike(n_knots=64, t0=W.T0_C1, max_batch=2)
    like.set_data(*data)
    assert LL.lisa_like_get_tune(like.h)[1] == 1
    assert same(like.loglike(th), want, dd)
    like.close()
    del hog
    torch.cuda.empty_cache()


def test_refused_data_leave_the_second_copy(pkg, orc):
    """Memory so short that an upload takes the second copy's room, and data that are refused
    then: the old data, and their copy, are in use as before."""
    import torch

    LL = pkg.lisalike
    n = 4000003
    data, th = problem(orc, n, 2)
    like = pkg.LisaLike(n_knots=64, t0=W.T0_C1, max_batch=2)
    like.set_data(*data)
    want = like.loglike(th)
    bad = data[4].copy()
    bad[1, n // 2] = 0.0
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - (72 * n + 36 * n), dtype=torch.uint8, device="cuda")
    with pytest.raises(pkg.lisalike.LisaError):
        like.set_data(*data[:4], bad)
    assert LL.lisa_like_get_tune(like.h)[1] == 8
    assert all(np.array_equal(x, y) for x, y in zip(like.loglike(th), want))
    like.close()
    del hog
    torch.cuda.empty_cache()
