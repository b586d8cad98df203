"""The chunked spline solve on few knots over four to six decades, where the second derivative
of the phase falls by many orders of magnitude from row to row and a short run-in would leave
a share of far rows in the near ones: every row of every series against the oracle's serial
solve of the device's own knot values.

Tolerance, row by row: with A M = rhs, rhs_i = 6 (slope_i - slope_{i-1}), the slopes carry a
relative rounding of 2 eps and their differences as much of the slopes (24 eps of |slope_i| + |slope_{i-1}|
with the factor 6 and twice for safety), an elimination without pivoting of a diagonally dominant matrix
8 eps |A| |M|, and |A^-1| takes both to M; the two sides are allowed that much each."""
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


def tolerance(x, y, M):
    n, eps = len(x), 2.0 ** -53
    h = np.diff(x)
    A = np.zeros((n - 2, n - 2))
    for i in range(1, n - 1):
        hp, hc = h[i - 1], h[i]
        row = {i - 1: hp, i: 2.0 * (hp + hc), i + 1: hc}
        if i == 1:
            row[i] += hp * (hp + hc) / hc
            row[i + 1] -= hp * hp / hc
        if i == n - 2:
            row[i] += hc * (hp + hc) / hp
            row[i - 1] -= hc * hc / hp
        for k, v in row.items():
            if 1 <= k <= n - 2:
                A[i - 1, k - 1] = v
    sl = np.abs(np.diff(y) / h)
    back = 24 * eps * (sl[1:] + sl[:-1]) + 8 * eps * (np.abs(A) @ np.abs(M))
    return 2.0 * (np.abs(np.linalg.inv(A)) @ back)


@pytest.mark.parametrize("B", [1, 40])  # one block a series; one block a system
@pytest.mark.parametrize("f0", [1e-6, 1e-5])
@pytest.mark.parametrize("K", [36, 40, 48, 66, 67, 128, 191, 192, 193])
def test_every_row(pkg, orc, K, f0, B):
    t0 = 1e13 if f0 == 1e-5 else 1e16  # the band begins near the first bin
    th = W.draw_walkers(B, 7, (3.0, 4.5))
    th[:, 4] = [orc.dl_gpc(z) for z in th[:, 4]]
    n = 2000
    like = pkg.LisaLike(modes=W.MODES6[:3], n_knots=K, t0=t0, max_batch=B)
    like.set_data(f0, 0.6 / n, n, None, np.ones((3, n)))
    band, fedge, fk, vals = like.stage_knots(th)
    coef = like.stage_coeffs(th)
    like.close()
    seen = 0
    for b, mi in ((0, 0), (B // 2, 1), (B - 1, 2)):
        if not band[b, mi, 0]:
            continue
        assert fedge[b, mi, 1] > (5e3 if f0 == 1e-5 else 5e4) * fedge[b, mi, 0]
        seen += 1
        for q in range(8):
            M = 2.0 * orc.spline(fk[b, mi], vals[b, mi, q])[1:, 2]  # rows 1 .. K - 2
            got = 2.0 * coef[b, mi, 1:, q, 2]
            tol = tolerance(fk[b, mi], vals[b, mi, q], M)
            worst = np.max(np.abs(got - M) / np.maximum(tol, 1e-300))
            assert worst <= 1.0, (b, mi, q, worst, int(np.argmax(np.abs(got - M) / np.maximum(tol, 1e-300))))
    assert seen
