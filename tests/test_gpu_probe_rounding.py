"""V_act is that of the gradients the sampled backward returns: the rows of kept data rescaled by 1/p and rounded to bf16
before the product.  All draws of a batch share p, so the rounding moves every value of a datum by the same factor, about
1e-4, which does not average out where a few data make up the sum or 1/p is near 1 (up to 5e-4 of V_act in these shapes).

Reference: the probe in float64 on rows rounded like that, at the library's own p.  Tolerance 5e-5: fp32 sums of up to 4400
products, 2e-6 of a gradient, whose difference from the exact one is at least a tenth of it, squared."""
import numpy as np
import pytest
import torch

from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import v_act_of_rounded_rows

pytestmark = pytest.mark.gpu


# one, two and eight steps of 64 rows per datum, remainders, sliced and whole tiles, two passes of draws, sampled columns
# (one and two batches at a time), data too short for the joint product (T < 64)
@pytest.mark.parametrize("N,T,d_in,d_out,M,rows", [(4, 64, 64, 64, 2, 0), (5, 197, 128, 192, 3, 0), (3, 130, 320, 448, 5, 0),
                                                   (8, 128, 64, 320, 2, 256), (4, 1100, 128, 256, 2, 64), (40, 72, 64, 128, 4, 64),
                                                   (3, 65, 1280, 1280, 2, 0), (6, 48, 64, 128, 3, 0)])
@pytest.mark.parametrize("rho", [0.8, 0.3])
def test_v_act_of_rounded_rows(N, T, d_in, d_out, M, rows, rho):
    vbuild.build()
    case = inputs.LayerCase("pr", N, T, d_in, d_out, torch.bfloat16, 0.3, 0.5, 0.5, 0.5)
    batches = [inputs.make_layer(case, batch=i) for i in range(M)]
    layer = vb.Layer(N, T, d_in, d_out, torch.bfloat16, vb.GEMM_TENSOR)
    if rows:
        layer.set_probe_subsample(rows, 9)
    Xs, dYs, W = [b[0].cuda() for b in batches], [b[1].cuda() for b in batches], batches[0][2].cuda()
    out = layer.variance_probe(Xs, dYs, W, rho, 0.5, 0.75, 42).cpu().numpy()
    ref = v_act_of_rounded_rows(layer, batches, rho, 42, layer.probe_subsample() if rows else None)
    assert out[1] == pytest.approx(ref, rel=5e-5)
    assert np.array_equal(layer.variance_probe(Xs, dYs, W, rho, 0.5, 0.75, 42).cpu().numpy(), out)
    assert layer.device_status() == 0
    layer.close()
