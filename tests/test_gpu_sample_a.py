"""SampleA over one to several data per lane and with sums by warps and by CTAs, few and more data than CTAs, with and without
partial sums and a list of alive data from the layer above: norms and probabilities within 1e-5 of the oracle (fp32 sums of up
to 70000 squares in a fixed tree), masks bit-exact for the returned probabilities, repeated calls bit-identical."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,parts", [(1, 5, 1), (32, 40, 1), (33, 1025, 1), (64, 30, 40), (65, 16, 1), (129, 9, 1), (257, 5, 300), (1024, 3, 1)])
def test_sample_a_from_handed_down_norms(N, T, parts):
    vbuild.build()
    d_in, d_out = 64, 64
    X, dY, W = inputs.make_layer(inputs.LayerCase("sa", N, T, d_in, d_out, torch.bfloat16, 1.0, 0.5, 0.5, 0.5))
    layer = vb.Layer(N, T, d_in, d_out, torch.bfloat16, vb.GEMM_TENSOR)
    Xc, dYc, Wc = X.cuda(), dY.cuda(), W.cuda()
    sq = (dYc.float() ** 2).sum(1)
    cut = torch.rand(N * T, parts, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) + 0.1
    a_in = (sq[:, None] * cut / cut.sum(1, keepdim=True)).contiguous()
    alive = torch.arange(0, N, 2, dtype=torch.int32, device="cuda")
    cnt = torch.tensor([len(alive)], dtype=torch.int32, device="cuda")
    dX, dW = torch.empty(N * T, d_in, dtype=torch.bfloat16, device="cuda"), torch.empty(d_out, d_in, device="cuda")
    for kw in ({}, dict(alive_in=alive, alive_cnt_in=cnt), dict(a_in=a_in, a_in_parts=parts, alive_in=alive, alive_cnt_in=cnt)):
        layer.linear_bwd_chain(Xc, dYc, Wc, 0.4, 0.5, 7, dX, dW, **kw)
        s = layer.last_sampling()
        G = np64(dY).reshape(N, T, d_out).copy()
        if kw:
            G[1::2] = 0.0
        g = np.sqrt((G ** 2).sum((1, 2)))
        assert np.allclose(np64(s.g), g, rtol=1e-5, atol=1e-30)
        assert np.allclose(np64(s.p), o.capped_prop(g, N * float(np.float32(0.4))), rtol=1e-5, atol=1e-12)
        keep = o.bernoulli_keep(s.p.cpu().numpy(), 7, 0)
        assert np.array_equal(s.idxA.cpu().numpy(), np.flatnonzero(keep))
        layer.linear_bwd_chain(Xc, dYc, Wc, 0.4, 0.5, 7, dX, dW, **kw)
        again = layer.last_sampling()
        assert torch.equal(again.g, s.g) and torch.equal(again.p, s.p) and torch.equal(again.idxA, s.idxA)
    assert layer.device_status() == 0
    layer.close()
