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


def test_long_contractions_do_not_drift():
    """Accumulation in TMEM truncates, 2^-25 of the sum per 16 rows on average: over the 32768 rows of these unsliced tiles V_s
    would lose 6e-5 (twice the gradient's share).  Sums of 1024 rows, added up in fp32, lose 2e-6 each: bound 1e-5."""
    vbuild.build()
    N, T, d_in, d_out = 16, 2048, 512, 4096
    case = inputs.LayerCase("pl", N, T, d_in, d_out, torch.bfloat16, 0.0, 1.0, 0.3, 0.3)
    batches = [inputs.make_layer(case, batch=b, device="cuda") for b in range(2)]
    layer = vb.Layer(N, T, d_in, d_out, torch.bfloat16, vb.GEMM_TENSOR)
    out = layer.variance_probe([b[0] for b in batches], [b[1] for b in batches], batches[0][2], 0.3, 0.5, 0.75, 42)
    G = [b[1].double().T @ b[0].double() for b in batches]
    assert float(out[0]) == pytest.approx(float(((G[0] - G[1]) ** 2).sum()) / 2, rel=1e-5)
    layer.close()
