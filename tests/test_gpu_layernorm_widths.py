"""LayerNorm behind SampleA at the widths where a row changes from one to sixteen warps and to the two-pass kernels, with few
and many rows, against the oracle.  Tolerances as derived for the narrower widths: one bf16 rounding of dX (2^-9 / sqrt(3) of its
norm) and fp32 sums; the column sums add up to 300 rows in fp32."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import f32, np64, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("N,T,d", [(1, 1, 8), (5, 60, 512), (5, 60, 520), (4, 33, 1024), (4, 33, 1032), (4, 33, 2000), (3, 21, 2056), (2, 9, 4096), (3, 21, 4104),
                                   (2, 9, 8192), (2, 9, 8200)])
def test_layernorm_bwd_at_every_row_group_size(dtype, N, T, d):
    vbuild.build()
    X, dY, _ = inputs.make_layer(inputs.LayerCase("ln", N, T, d, d, dtype, 0.5, 0.5, 0.5, 0.5), d_out=d)
    X = (X.float() * 1.3 - 0.4).to(dtype)
    gamma = (1.0 + 0.2 * torch.randn(d, generator=torch.Generator().manual_seed(5))).to(dtype)
    layer = vb.Layer(N, T, d, d, dtype, vb.GEMM_FMA)
    a_out = torch.full((N * T, layer.chain_parts()), 7.0, device="cuda")
    args = (X.cuda(), gamma.cuda(), dY.cuda())
    dX, dg, db = layer.layernorm_bwd(*args, 0.6, 3, a_out=a_out)
    s = layer.last_sampling()
    ref = o.layernorm_bwd(np64(X), np64(gamma), np64(dY), N, T, f32(0.6), 3, p_override=s.p.cpu().numpy())
    tol = 2.5e-3 if dtype == torch.bfloat16 else 2e-5
    assert rel_fro(np64(dX), ref["dX"]) <= tol
    assert rel_fro(np64(dg), ref["dgamma"]) <= 2e-5 and rel_fro(np64(db), ref["dbeta"]) <= 2e-5
    assert np.allclose(np64(a_out).sum(axis=1), (np64(dX) ** 2).sum(axis=1), rtol=1e-5, atol=1e-30)
    again = layer.layernorm_bwd(*args, 0.6, 3)
    assert torch.equal(dX, again[0]) and torch.equal(dg, again[1]) and torch.equal(db, again[2])
    layer.close()
