"""The weight of an fp32 layer cut while SampleA runs, on both sides of the line (14 GFLOP of part products) and with widths that
leave pieces over: bit for bit the outputs of the same call with stage profiling, which runs the stages one after the other, with
another weight in every call."""
import pytest
import torch

from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,d_in,d_out,rho", [(16, 128, 768, 3072, 0.5), (40, 100, 776, 1032, 0.36), (40, 100, 776, 1032, 0.37),
                                                (3, 700, 2056, 520, 1.0), (128, 128, 256, 272, 1.0)])
def test_same_as_one_after_the_other(N, T, d_in, d_out, rho):
    vbuild.build()
    dtype = torch.float32
    X, dY, W = (t.cuda() for t in inputs.make_layer(inputs.LayerCase("se", N, T, d_in, d_out, dtype, 1.0, 0.5, rho, 0.5)))
    beside, alone = vb.Layer(N, T, d_in, d_out, dtype), vb.Layer(N, T, d_in, d_out, dtype)
    alone.set_profiling(True)
    for i in range(4):
        Wi = W * (1.0 + i)
        a, b = beside.linear_bwd(X, dY, Wi, rho, 0.5, 3 + i), alone.linear_bwd(X, dY, Wi, rho, 0.5, 3 + i)
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        assert float(a[0].abs().max()) > 0.0
    assert beside.device_status() == 0 and alone.device_status() == 0
    beside.close(); alone.close()
