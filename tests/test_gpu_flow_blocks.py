"""The flow's kernels at the edges of their blocks of 16 samples and of the 2048 samples whose
weight-gradient operands are held at a time."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle_flow as F
from test_gpu_flow import D, pkg, setup_flow  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 250])
def test_a_row_does_not_depend_on_its_neighbours(pkg, n):  # noqa: F811
    rng, mu, sig, w, fl = setup_flow(pkg, 11, 0.2)
    x = mu + sig * rng.normal(size=(300, D))
    for run in (fl.normalize, fl.generate):
        y, lq = run(x)
        for first in (0, 7):
            ys, lqs = run(x[first:first + n])
            assert np.array_equal(ys, y[first:first + n]) and np.array_equal(lqs, lq[first:first + n])
    fl.close()


@pytest.mark.parametrize("n", [64, 2048, 2112])
def test_gradients_over_the_held_samples(pkg, n):  # noqa: F811
    """Tolerances of the gradient test of 512 samples (bfloat16 operands on both sides)."""
    rng, mu, sig, w, fl = setup_flow(pkg, 5, 0.2)
    x = mu + sig * rng.normal(size=(n, D))
    loss, g = fl.gradients(x)
    want, ref = F.nll_grads(w, F.whiten(x, mu, sig))
    assert abs(loss - want) <= 1e-4 * max(1.0, abs(want))
    for k in g:
        assert np.linalg.norm(g[k] - ref[k]) <= 2e-2 * max(np.linalg.norm(ref[k]), 1e-30), k
    fl.close()


@pytest.mark.parametrize("batch", [64, 2112])
def test_training_repeats_and_follows_the_oracle(pkg, batch):  # noqa: F811
    import torch

    data = np.random.default_rng(2).normal(size=(5000, D)) @ np.diag(np.linspace(0.5, 2.0, D))
    w0 = W.flow_init_weights(3, 0.0)
    out = []
    for _ in range(2):
        fl = pkg.lisalike.Flow(seed=1)
        fl.set_weights(w0)
        out.append((fl.train(torch.tensor(data, device="cuda"), 4, batch=batch, lr=1e-3, seed=7), fl.weights()))
        fl.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert all(np.array_equal(out[0][1][k], out[1][1][k]) for k in out[0][1])
    losses = F.train(w0, data, 4, batch, 1e-3, F.minibatch_index(7))[3]
    # losses of about 10; the first steps move every weight by lr whatever the gradient's
    # rounding, so they agree to a bfloat16 step of the outputs
    assert np.max(np.abs(out[0][0] - losses)) <= 1e-2
