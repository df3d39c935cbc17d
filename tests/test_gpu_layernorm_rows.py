"""LayerNorm behind SampleA with several rows per row group (each loaded while the one before is worked on), at the widths of the
groups of one to sixteen warps, dropped rows written or left.  Tolerances: one bf16 rounding of dX (2^-9 / sqrt(3) of its norm) and
fp32 sums; the column sums add up to 6000 rows in fp32, in a tree of row groups, CTAs and ranges of them."""
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
@pytest.mark.parametrize("N,T,d", [(30, 200, 256), (30, 200, 264), (7, 857, 768), (30, 100, 776), (2500, 2, 64), (30, 200, 512),
                                   (25, 100, 1032), (9, 200, 1544), (10, 100, 2000), (42, 100, 2000), (9, 100, 2056), (9, 100, 4096),
                                   (21, 100, 4096), (9, 100, 4104)])
def test_rows_loaded_ahead(dtype, N, T, d):
    vbuild.build()
    X, dY, _ = inputs.make_layer(inputs.LayerCase("ln", N, T, d, d, dtype, 0.5, 0.5, 0.5, 0.5), d_out=d)
    X = (X.float() * 1.3 - 0.4).to(dtype)
    gamma = (1.0 + 0.2 * torch.randn(d, generator=torch.Generator().manual_seed(5))).to(dtype)
    layer = vb.Layer(N, T, d, d, dtype)
    args = (X.cuda(), gamma.cuda(), dY.cuda())
    dX, dg, db = layer.layernorm_bwd(*args, 0.7, 3)
    s = layer.last_sampling()
    ref = o.layernorm_bwd(np64(X), np64(gamma), np64(dY), N, T, f32(0.7), 3, p_override=s.p.cpu().numpy())
    assert rel_fro(np64(dX), ref["dX"]) <= (2.5e-3 if dtype == torch.bfloat16 else 2e-5)
    assert rel_fro(np64(dg), ref["dgamma"]) <= 2e-5 and rel_fro(np64(db), ref["dbeta"]) <= 2e-5
    # dropped rows are left alone where the caller says so, the others do not change
    kept = torch.zeros(N, dtype=torch.bool, device="cuda")
    kept[s.idxA.long()] = True
    rows = kept.repeat_interleave(T)
    assert not dX[~rows].any()
    other = torch.full_like(dX, 7.0)
    layer.layernorm_bwd(*args, 0.7, 3, dX=other, skip_dropped_rows=True)
    assert torch.equal(other[rows], dX[rows]) and bool((other[~rows] == 7.0).all())
    layer.close()
