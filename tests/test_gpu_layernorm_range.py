"""LayerNorm of activations and gradients far from 1: products of a row's statistics must not leave fp32's range where the result
does not (1/sigma squared times a mean of the gradient does: 1e-44 for x of 1e17 and dY of 1e-10, 1e39 for 1e-18 and 1e5).
Tolerances as derived for ordinary values: one bf16 rounding of dX (2^-9 / sqrt(3) of its norm) and fp32 sums."""
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import f32, np64, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("N,T,d", [(6, 50, 512), (4, 33, 1032)])
@pytest.mark.parametrize("x,y,eps", [(1e17, 1e-10, 1e-5), (1e-18, 1e5, 0.0)])
def test_values_far_from_one(dtype, N, T, d, x, y, eps):
    vbuild.build()
    X, dY, _ = inputs.make_layer(inputs.LayerCase("ln", N, T, d, d, dtype, 0.5, 0.5, 0.5, 0.5), d_out=d)
    X, dY = ((X.float() * 1.3 - 0.4) * x).to(dtype), (dY.float() * y).to(dtype)
    gamma = (1.0 + 0.2 * torch.randn(d, generator=torch.Generator().manual_seed(5))).to(dtype)
    layer = vb.Layer(N, T, d, d, dtype)
    dX, dg, db = layer.layernorm_bwd(X.cuda(), gamma.cuda(), dY.cuda(), 0.7, 3, eps=eps)
    p = layer.last_sampling().p.cpu().numpy()
    ref = o.layernorm_bwd(np64(X), np64(gamma), np64(dY), N, T, f32(0.7), 3, eps=f32(eps), p_override=p)
    assert rel_fro(np64(dX), ref["dX"]) <= (2.5e-3 if dtype == torch.bfloat16 else 2e-5)
    assert rel_fro(np64(dg), ref["dgamma"]) <= 2e-5 and rel_fro(np64(db), ref["dbeta"]) <= 2e-5
    layer.close()
