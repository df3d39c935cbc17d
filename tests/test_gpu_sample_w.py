"""SampleW's single-CTA stage at the edges of its register variants (2, 4, 8 and 16 scores a thread of 1024) and of its chunks of
32 rows: kept-row lists, their ends and the probabilities against the oracle, on the rows of a few large data and of many small
ones, with a budget that covers every score (q = 1) and one that does not."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T", [(1, 31), (1, 1024), (2, 1024), (3, 683), (4, 1024), (241, 17), (8, 1024), (5, 1639), (16, 1024),
                                 (4, 4097), (1021, 3)])
@pytest.mark.parametrize("rho,nu", [(1.0, 0.3), (0.6, 1.0)])
def test_rows_kept_at_the_edges(N, T, rho, nu):
    vbuild.build()
    case = inputs.LayerCase("w", N, T, 64, 64, torch.float32, 0.5, 1.0, rho, nu)
    X, dY, W = inputs.make_layer(case)
    layer = vb.Layer(N, T, 64, 64, torch.float32)
    s = layer.score(X.cuda(), dY.cuda(), rho, nu, 5)
    ref = o.linear_bwd(np64(X), np64(dY), np64(W), N, T, float(np.float32(rho)), float(np.float32(nu)), 5)
    assert np.array_equal(s.idxA.cpu().numpy(), ref["idxA"])
    q, idx = s.q.cpu().numpy().astype(np.float64), s.idxW.cpu().numpy()
    # fp32 tree sums of up to 16384 non-negative scores against float64: 2e-5, the bound the probabilities are specified to
    assert np.abs(q - ref["q32"]).max() <= 2e-5 * max(1.0, np.abs(ref["q32"]).max())
    # given these probabilities the list is that of the uniforms, in ascending order, bit for bit
    keep = o.bernoulli_keep(s.q.cpu().numpy(), 5, 1) & np.repeat(np.isin(np.arange(N), ref["idxA"]), T)
    assert np.array_equal(idx, np.flatnonzero(keep)) and s.cntW == idx.size
    assert layer.device_status() == 0
    layer.close()
