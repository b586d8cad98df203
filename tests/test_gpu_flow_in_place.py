"""The flow's two directions with the output written over the input, at row counts around a
block's 16: the same bits as with an output of its own."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 300])
def test_output_over_the_input(n):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2005_01827_gb300 import build

    build.build()
    from paper_2005_01827_gb300 import lisalike as LL

    fl = LL.Flow(3)
    fl.set_weights(W.flow_init_weights(5, 0.3))
    lib = LL.load()
    x = torch.randn((n, 11), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(n))
    for call in (lib.lisa_flow_generate, lib.lisa_flow_normalize):
        out, both = torch.empty_like(x), x.clone()
        q = torch.empty((2, n), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert call(fl.h, LL._ptr(x), n, LL._ptr(out), LL._ptr(q[0]), None) == 0
        assert call(fl.h, LL._ptr(both), n, LL._ptr(both), LL._ptr(q[1]), None) == 0
        torch.cuda.synchronize()
        assert torch.equal(out, both) and torch.equal(q[0], q[1])
    fl.close()
