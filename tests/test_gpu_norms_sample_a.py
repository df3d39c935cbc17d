"""Row norms and SampleA at the edges of their common launch (32 data, 3200 rows, sums of 1024): the data's norms are those of the
two launches bit for bit (a layer of more data that begins with the same ones takes these), the probabilities within 1e-5 of the
oracle (fp32 sums in fixed trees), the masks exact for them; lists of alive data, their bad entries and lengths."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("N,T,d_out", [(1, 1, 64), (3, 1024, 72), (3, 1025, 64), (32, 100, 64), (31, 103, 200), (33, 33, 64), (32, 101, 64),
                                       (7, 131, 8)])
def test_one_launch_and_two(N, T, d_out, dtype):
    vbuild.build()
    d_in, M = 64, max(N, 33)
    X, dY, W = (t.cuda() for t in inputs.make_layer(inputs.LayerCase("ns", M, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5)))
    alive = torch.arange(0, N, 2, dtype=torch.int32, device="cuda").flip(0).contiguous()
    bad = alive.clone()
    bad[0] = N
    i32 = lambda v: torch.tensor([v], dtype=torch.int32, device="cuda")
    listed = np.arange(N) % 2 == 0
    unbad = listed.copy()
    unbad[bad.numel() * 2 - 2] = False
    lists = [({}, np.ones(N, bool), 0), (dict(alive_in=alive, alive_cnt_in=i32(alive.numel())), listed, 0),
             (dict(alive_in=bad, alive_cnt_in=i32(bad.numel())), unbad, -1),
             (dict(alive_in=alive, alive_cnt_in=i32(-1)), np.zeros(N, bool), -1)]
    for kw, mask, status in lists:
        norms = []
        for n in (N, M):
            layer = vb.Layer(n, T, d_in, d_out, dtype)
            dX, dW = torch.empty(n * T, d_in, dtype=dtype, device="cuda"), torch.empty(d_out, d_in, device="cuda")
            if n != N and kw and status:
                layer.close()
                continue      # another N: other entries are bad
            for _ in range(2):
                layer.linear_bwd_chain(X[:n * T], dY[:n * T], W, 0.4, 0.5, 7, dX, dW, **kw)
                s = layer.last_sampling()
                norms.append(s.g[:N].clone())
                assert layer.device_status() == (status if n == N else 0)
            if n == N:
                p, idx = s.p.cpu().numpy(), s.idxA.cpu().numpy()
            layer.close()
        assert all(torch.equal(g, norms[0]) for g in norms)
        G = np64(dY[:N * T]).reshape(N, T, d_out) * mask[:, None, None]
        g = np.sqrt((G ** 2).sum((1, 2)))
        assert np.allclose(np64(norms[0]), g, rtol=1e-5, atol=1e-30)
        assert np.allclose(p, o.capped_prop(g, N * float(np.float32(0.4))), rtol=1e-5, atol=1e-12)
        assert np.array_equal(idx, np.flatnonzero(o.bernoulli_keep(p, 7, 0)))
