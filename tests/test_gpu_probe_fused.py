"""The probe with one product launch for the exact gradients and all draws, against the oracle: one to several k-blocks per
datum with and without remainders (of 64 and of 16 rows), tiles past d_out, sliced and whole tiles, more tiles than SMs, two
to five draws (one and two rounds of accumulators), many data, and the sample of the parameters.

Tolerances: V_s and V_act carry fp32 sums (1e-4 of float64, as for the fp32 path: differences of sums of up to 16000 terms,
1e-5 each), V_act on the rows as they enter the product, rounded to bf16; V_w fp32 water-filling (1e-4), p_lo and p_hi are
exact."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import f32, np64, v_act_of_rounded_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,d_in,d_out,M,rows", [(4, 64, 64, 64, 2, 0), (5, 197, 128, 192, 3, 0), (3, 130, 320, 448, 5, 0),
                                                   (40, 72, 64, 128, 4, 64), (2, 1100, 128, 256, 2, 128),
                                                   (3, 65, 1280, 1280, 2, 0)])
def test_fused_probe_matches_oracle(N, T, d_in, d_out, M, rows):
    vbuild.build()
    case = inputs.LayerCase("pf", N, T, d_in, d_out, torch.bfloat16, 1.0, 0.5, 0.5, 0.5)
    batches = [inputs.make_layer(case, batch=i) for i in range(M)]
    cfg = vb.default_config()
    cfg.alpha = 0.05
    layer = vb.Layer(N, T, d_in, d_out, torch.bfloat16, vb.GEMM_TENSOR, cfg)
    if rows:
        layer.set_probe_subsample(rows, 9)
    Xs, dYs, W = [b[0].cuda() for b in batches], [b[1].cuda() for b in batches], batches[0][2].cuda()
    run = lambda: layer.variance_probe(Xs, dYs, W, 0.4, 0.5, 0.75, 42).cpu().numpy()
    out = run()
    ref = o.variance_probe([np64(b[0]) for b in batches], [np64(b[1]) for b in batches], np64(batches[0][2]), N, T, f32(0.4), 0.5,
                           s=0.75, alpha=f32(0.05), seed=42, param_rows=layer.probe_subsample() if rows else None)
    v_act = v_act_of_rounded_rows(layer, batches, 0.4, 42, layer.probe_subsample() if rows else None)
    assert out[0] == pytest.approx(ref["V_s"], rel=1e-4) and out[1] == pytest.approx(v_act, rel=1e-4)
    assert out[2] == pytest.approx(ref["V_w"], rel=1e-4)
    assert out[3] == pytest.approx(ref["p_lo"], abs=1e-6) and out[4] == pytest.approx(ref["p_hi"], abs=1e-6)
    assert np.array_equal(run(), out)
    # a sampled call in between shares the workspace
    layer.linear_bwd(Xs[0], dYs[0], W, 0.5, 0.5, 1)
    assert np.array_equal(run(), out) and layer.device_status() == 0
    # a wait that runs out is reported and the handle recovers
    layer.set_wait_limit(2_000_000, stall_once=True)
    run()
    assert layer.device_status() == -6
    layer.set_wait_limit(2_000_000_000, stall_once=False)
    assert np.array_equal(run(), out) and layer.device_status() == 0
    # captured in a graph with its scoring a batch ahead on the handle's own stream
    got = torch.zeros(5, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        layer.variance_probe(Xs, dYs, W, 0.4, 0.5, 0.75, 42, out=got)
    g.replay()
    assert np.array_equal(got.cpu().numpy(), out)
    del g
    layer.close()


@pytest.mark.parametrize("d_out,rows", [(2048, 64), (2112, 256), (4160, 192), (6208, 64)])
def test_sampled_columns_over_several_chunks_of_a_row(d_out, rows):
    """The columns are picked 2048 at a time, 32 per step: one to eight steps in a chunk, a last chunk of 64."""
    vbuild.build()
    N, T, d_in, M = 3, 64, 64, 2
    case = inputs.LayerCase("pc", N, T, d_in, d_out, torch.bfloat16, 1.0, 0.5, 0.5, 0.5)
    batches = [inputs.make_layer(case, batch=i) for i in range(M)]
    layer = vb.Layer(N, T, d_in, d_out, torch.bfloat16, vb.GEMM_TENSOR)
    layer.set_probe_subsample(rows, 3)
    out = layer.variance_probe([b[0].cuda() for b in batches], [b[1].cuda() for b in batches], batches[0][2].cuda(), 0.4, 0.5,
                               0.75, 42).cpu().numpy()
    ref = o.variance_probe([np64(b[0]) for b in batches], [np64(b[1]) for b in batches], np64(batches[0][2]), N, T, f32(0.4), 0.5,
                           s=0.75, alpha=0.05, seed=42, param_rows=layer.probe_subsample())
    v_act = v_act_of_rounded_rows(layer, batches, 0.4, 42, layer.probe_subsample())
    assert out[:3] == pytest.approx([ref["V_s"], v_act, ref["V_w"]], rel=1e-4)
    layer.close()
