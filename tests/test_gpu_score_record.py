"""The record that a scoring call writes as it emits the kept rows: the same, bit for bit, as the one copied from the workspace
afterwards and as that of the call without a handle, at the edges of its chunks of 32 rows and CTAs of 256, with data of few and
many rows, nothing dropped and most dropped; outputs not asked for are not written, and alter no other."""
import ctypes as C

import pytest
import torch

from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs

pytestmark = pytest.mark.gpu
NAMES = ("g", "p", "w", "q", "idxA", "cntA", "idxW", "cntW")


@pytest.mark.parametrize("N,T,dtype", [(1, 1, torch.float32), (1, 31, torch.bfloat16), (3, 11, torch.float32), (4, 64, torch.bfloat16),
                                       (257, 1, torch.float32), (1100, 3, torch.bfloat16), (5, 1639, torch.bfloat16), (9, 2048, torch.float32)])
@pytest.mark.parametrize("rho,nu", [(1.0, 1.0), (0.15, 0.5)])
def test_record_written_and_copied(N, T, dtype, rho, nu):
    vbuild.build()
    R, d = N * T, 64
    X, dY, _ = (t.cuda() for t in inputs.make_layer(inputs.LayerCase("sr", N, T, d, d, dtype, 0.5, 1.0, rho, nu)))
    layer = vb.Layer(N, T, d, d, dtype)
    got = [layer.score(X, dY, rho, nu, 5), layer.last_sampling()]
    if R <= 16384 and N <= 4096:
        got.append(vb.score_static(X, dY, N, T, rho, nu, 5))
    for s in got[1:]:
        for name in NAMES:
            a, b = getattr(got[0], name), getattr(s, name)
            assert torch.equal(a, b) if torch.is_tensor(a) else a == b, name
    out = dict(zip(NAMES, [torch.full((n,), -7, device="cuda", dtype=t) for n, t in
                           zip((N, N, R, R, N, 1, R, 1), [torch.float32] * 4 + [torch.int32] * 4)]))
    for skip in (0, 1):
        ptr = [C.c_void_p(out[n].data_ptr() if i % 2 == skip else 0) for i, n in enumerate(NAMES)]
        f = vb.lib().vcas_score
        rc = f(layer._h, vb._ptr(X), vb._ptr(dY), rho, nu, 5, *ptr, vb._stream())
        assert rc == 0
        for i, n in enumerate(NAMES):
            if i % 2 != skip:
                assert skip == 1 or bool((out[n] == -7).all()), n
                continue
            ref = getattr(got[0], n)
            assert torch.equal(out[n][:ref.numel()], ref) if torch.is_tensor(ref) else int(out[n]) == ref, n
    assert layer.device_status() == 0
    layer.close()
