"""The calls around the split products (fp32 layers, and bf16 widths that are not multiples of 64): probe, sample of the
parameters, chain with its lists and deferred join, stage profiling, a wait that runs out in a sampled call.

Tolerances: products within 1e-6 of fp32 arithmetic in another order (see test_gpu_split.py), a bf16 dX one rounding, so that a
value in thousands falls on the other side (1e-3); the probe as the fp32 path (differences of sums, 1e-4)."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import f32, np64, rel_fro

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


# odd draws use the second workspace set, whose operands share memory with the first's; few tiles: sliced contractions, and one
# slice (a contraction of 3 x 16 rows)
@pytest.mark.parametrize("dtype,N,T,d_in,d_out,M,rows", [(F32, 8, 40, 64, 136, 3, 0), (F32, 5, 130, 200, 72, 4, 0), (F32, 8, 48, 128, 136, 3, 40),
                                                         (F32, 4, 200, 128, 512, 3, 256), (BF16, 8, 40, 72, 136, 3, 0),
                                                         (BF16, 5, 130, 200, 72, 4, 0), (BF16, 8, 48, 120, 136, 3, 8), (F32, 3, 16, 8, 8, 2, 0)])
def test_probe_matches_oracle(dtype, N, T, d_in, d_out, M, rows):
    vbuild.build()
    case = inputs.LayerCase("sp", N, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5)
    batches = [inputs.make_layer(case, batch=i) for i in range(M)]
    cfg = vb.default_config()
    cfg.alpha = 0.05
    layer = vb.Layer(N, T, d_in, d_out, dtype, vb.GEMM_AUTO, cfg)
    if rows:
        layer.set_probe_subsample(rows, 7)
    Xs, dYs, W = [b[0].cuda() for b in batches], [b[1].cuda() for b in batches], batches[0][2].cuda()
    run = lambda: layer.variance_probe(Xs, dYs, W, 0.4, 0.5, 0.75, 42).cpu().numpy()
    out = run()
    ref = o.variance_probe([np64(b[0]) for b in batches], [np64(b[1]) for b in batches], np64(batches[0][2]), N, T, f32(0.4), 0.5,
                           s=0.75, alpha=f32(0.05), seed=42, param_rows=layer.probe_subsample() if rows else None)
    assert out[:3] == pytest.approx([ref["V_s"], ref["V_act"], ref["V_w"]], rel=1e-4)
    assert out[3:] == pytest.approx([ref["p_lo"], ref["p_hi"]], abs=1e-6)
    layer.linear_bwd(Xs[0], dYs[0], W, 0.5, 0.5, 1)      # shares the workspace
    assert np.array_equal(run(), out) and layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("dtype,N,T,d_in,d_out", [(F32, 6, 50, 72, 200), (F32, 20, 33, 264, 72), (BF16, 6, 50, 72, 200), (BF16, 9, 140, 264, 520)])
def test_chain_matches_the_fma_products(dtype, N, T, d_in, d_out):
    """The same chain calls on a handle with split products and on one with FMA products, whose scoring is the same: lists and
    sampling records equal, outputs within the tolerance."""
    vbuild.build()
    X, dY, W = [t.cuda() for t in inputs.make_layer(inputs.LayerCase("c", N, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5))]
    H = torch.randn(N * T, d_in, generator=torch.Generator("cuda").manual_seed(3), device="cuda").to(dtype)
    alive = torch.arange(0, N, 2, dtype=torch.int32, device="cuda")
    cnt = torch.tensor([len(alive)], dtype=torch.int32, device="cuda")
    a_in = (dY.float() ** 2).sum(1)
    got = []
    for path in (vb.GEMM_AUTO, vb.GEMM_FMA):
        layer = vb.Layer(N, T, d_in, d_out, dtype, path)
        res = []
        for defer in (False, True):
            dX, dW = torch.full((N * T, d_in), 7.0, dtype=dtype, device="cuda"), torch.full((d_out, d_in), 7.0, device="cuda")
            a_out = torch.full((N * T, layer.chain_parts()), 7.0, device="cuda")
            kept, kept_cnt = torch.zeros(N, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
            layer.linear_bwd_chain(X, dY, W, 0.5, 0.5, 9, dX, dW, H=H, a_in=a_in, a_in_parts=1, alive_in=alive, alive_cnt_in=cnt,
                                   a_out=a_out, kept_out=kept, kept_cnt_out=kept_cnt, skip_dropped_rows=True, defer_join=defer)
            if defer:
                layer.join()
            s = layer.last_sampling()
            res.append((np64(dX), np64(dW), np64(a_out), kept[: int(kept_cnt)].tolist(), s.idxW.tolist(), s.p, s.q))
        for x, y in zip(res[0], res[1]):
            assert np.array_equal(np.asarray(x.cpu() if torch.is_tensor(x) else x), np.asarray(y.cpu() if torch.is_tensor(y) else y))
        assert layer.device_status() == 0
        layer.close()
        got.append(res[0])
    (dXa, dWa, aa, ka, ia, pa, qa), (dXb, dWb, _, kb, ib, pb, qb) = got
    assert ka == kb and ia == ib and torch.equal(pa, pb) and torch.equal(qa, qb) and set(ka) <= set(alive.tolist())
    assert rel_fro(dXa, dXb) <= (1e-6 if dtype == F32 else 1e-3) and rel_fro(dWa, dWb) <= 1e-6
    assert np.allclose(aa.sum(1), (dXa ** 2).sum(1), rtol=1e-5, atol=1e-30)
    dropped = [n for n in range(N) if n not in ka]
    assert not dXa.reshape(N, T, -1)[dropped].any()          # this path writes the rows of dropped data


@pytest.mark.parametrize("dtype,N,T,d_in,d_out", [(F32, 6, 50, 72, 200), (BF16, 6, 50, 72, 200), (F32, 33, 150, 776, 1000)])
def test_profiled_and_timed_out_sampled_calls(dtype, N, T, d_in, d_out):
    vbuild.build()
    X, dY, W = [t.cuda() for t in inputs.make_layer(inputs.LayerCase("c", N, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5))]
    layer = vb.Layer(N, T, d_in, d_out, dtype)
    dX, dW = layer.linear_bwd(X, dY, W, 0.5, 0.5, 9)
    dXd, dWd = layer.dense_bwd(X, dY, W)
    layer.set_profiling(True)                                 # one stream, a stage after the other
    pX, pW = layer.linear_bwd(X, dY, W, 0.5, 0.5, 9)
    pXd, pWd = layer.dense_bwd(X, dY, W)
    ms, calls = layer.stage_times()
    layer.set_profiling(False)
    assert list(calls) == [1, 1] and all(t > 0 for t in ms[:7])
    assert torch.equal(pX, dX) and torch.equal(pW, dW) and torch.equal(pXd, dXd) and torch.equal(pWd, dWd)
    layer.set_wait_limit(2_000_000, stall_once=True)
    layer.linear_bwd(X, dY, W, 0.5, 0.5, 9)
    assert layer.device_status() == -6
    layer.set_wait_limit(2_000_000_000, stall_once=False)
    again = layer.linear_bwd(X, dY, W, 0.5, 0.5, 9)
    assert torch.equal(again[0], dX) and torch.equal(again[1], dW) and layer.device_status() == 0
    layer.close()
