"""Products with operands cut into bf16 parts: fp32 layers, and bf16 layers whose widths are not multiples of 64.

Tolerances: fp32 results within 1e-6 of the float64 oracle (the parts are exact, products below 2^-26 are left out,
sums of a stage of 32 or 64 terms are truncated to 24 bits and added up in fp32: measured below 4e-7); a bf16 layer's dW,
whose rescaled rows are not rounded to bf16, meets the same, its dX carries one bf16 rounding (2^-9 / sqrt(3) of its norm)."""
import numpy as np
import pytest
import torch

from oracle import vcas_oracle as o
from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs
from tests.util import np64, rel_fro

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


# one row, one k-block, tiles that span data (T below and above 128, not dividing it), ragged widths, contractions cut
# into slices (few tiles, many k-blocks), more tiles than SMs
@pytest.mark.parametrize("shape", [(1, 1, 8, 8), (4, 64, 256, 256), (3, 50, 72, 200), (5, 197, 128, 1000), (2, 130, 64, 4096),
                                   (16, 256, 72, 64), (33, 150, 776, 1000), (9, 333, 1032, 520), (40, 128, 1288, 72)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_split_products_match_oracle(dtype, shape):
    vbuild.build()
    N, T, d_in, d_out = shape
    if dtype == BF16 and d_in % 64 == 0 and d_out % 64 == 0:
        d_out += 8                                     # multiples of 64 take the other tensor-core kernels
    X, dY, W = inputs.make_layer(inputs.LayerCase("t", N, T, d_in, d_out, dtype, 1.5, 1.0, 0.5, 0.5))
    H = (2.0 * torch.randn(N * T, d_in, generator=torch.Generator().manual_seed(3))).to(dtype)
    layer = vb.Layer(N, T, d_in, d_out, dtype)
    Xc, dYc, Wc, Hc = [t.cuda() for t in (X, dY, W, H)]
    gp = o.gelu_prime(np64(H))
    tol_x, tol_w = (1e-6 if dtype == F32 else 2.5e-3), 1e-6
    for seed, rho, nu in [(3, 0.5, 0.5), (11, 0.3, 0.4), (5, 1.0, 1.0)]:
        ref = o.linear_bwd(np64(X), np64(dY), np64(W), N, T, rho, nu, seed)
        p_in, q_in = torch.from_numpy(ref["p32"]).cuda(), torch.from_numpy(ref["q32"]).cuda()
        dX, dW = layer.linear_bwd(Xc, dYc, Wc, rho, nu, seed, p_in=p_in, q_in=q_in, H=Hc)
        assert rel_fro(np64(dX), ref["dX"] * gp) <= tol_x and rel_fro(np64(dW), ref["dW"]) <= tol_w
        assert not np64(dX)[~ref["keepA"].repeat(T)].any()
        again = layer.linear_bwd(Xc, dYc, Wc, rho, nu, seed, p_in=p_in, q_in=q_in, H=Hc)
        assert torch.equal(dX, again[0]) and torch.equal(dW, again[1])
    dXd, dWd = o.dense_bwd(np64(X), np64(dY), np64(W))
    dX, dW = layer.dense_bwd(Xc, dYc, Wc)
    assert rel_fro(np64(dX), dXd) <= tol_x and rel_fro(np64(dW), dWd) <= tol_w
    assert layer.device_status() == 0
    # a wait that runs out is reported and the handle recovers
    layer.set_wait_limit(2_000_000, stall_once=True)
    layer.dense_bwd(Xc, dYc, Wc)
    assert layer.device_status() == -6
    layer.set_wait_limit(2_000_000_000, stall_once=False)
    again = layer.dense_bwd(Xc, dYc, Wc)
    assert torch.equal(dX, again[0]) and torch.equal(dW, again[1]) and layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 3.4e38])
def test_split_products_of_values_without_a_finite_bf16_part(value):
    """An infinite or NaN weight, or one whose products overflow, leaves only its own column not finite."""
    vbuild.build()
    N, T, d_in, d_out = 2, 40, 72, 64
    X, dY, W = inputs.make_layer(inputs.LayerCase("t", N, T, d_in, d_out, F32, 1.0, 0.5, 0.5, 0.5))
    dY, W = dY.abs() + 0.5, W.clone()
    W[5, 7] = value
    layer = vb.Layer(N, T, d_in, d_out, F32)
    dX, dW = layer.dense_bwd(X.cuda(), dY.cuda(), W.cuda())
    col = dX[:, 7].cpu()
    if value != value:
        assert torch.isnan(col).all()
    else:
        assert (torch.isinf(col) | (col > 1e37)).all()
    keep = [c for c in range(d_in) if c != 7]
    ref = np64(dY) @ np64(W)[:, keep]
    assert rel_fro(np64(dX[:, keep]), ref) <= 1e-6
    layer.close()


@pytest.mark.parametrize("dtype", [F32, BF16])
@pytest.mark.parametrize("which", ["W", "H", "dX", "dW"])
def test_tensors_off_16_byte_boundaries(dtype, which):
    """Layers on this path take tensors that start on any element, views into flat buffers for instance: same results (fp32
    sums of up to 200 terms in another order, 1e-6; bf16 dX one rounding, as above)."""
    vbuild.build()
    N, T, d_in, d_out = 4, 50, 72, 200
    X, dY, W = [t.cuda() for t in inputs.make_layer(inputs.LayerCase("t", N, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5))]
    H = torch.randn(N * T, d_in, generator=torch.Generator("cuda").manual_seed(3), device="cuda").to(dtype)
    dX, dW = torch.empty(N * T, d_in, dtype=dtype, device="cuda"), torch.empty(d_out, d_in, device="cuda")
    t = dict(W=W, H=H, dX=dX, dW=dW)
    off = dict(t)
    flat = torch.empty(t[which].numel() + 1, dtype=t[which].dtype, device="cuda")
    off[which] = flat[1:].view(t[which].shape).copy_(t[which])
    layer = vb.Layer(N, T, d_in, d_out, dtype)
    def run(k, sampled):
        k["dX"].zero_(), k["dW"].zero_()
        if sampled:
            layer.linear_bwd(X, dY, k["W"], 0.6, 0.5, 3, H=k["H"], dX=k["dX"], dW=k["dW"])
        else:
            layer.dense_bwd(X, dY, k["W"], H=k["H"], dX=k["dX"], dW=k["dW"])
        return np64(k["dX"]), np64(k["dW"])
    for sampled in (True, False):
        (rX, rW), (gX, gW) = run(t, sampled), run(off, sampled)
        # a bf16 layer's dX rounds sums that differ by 1e-7 of themselves: one value in thousands falls on the other side
        assert rel_fro(gX, rX) <= (1e-6 if dtype == F32 else 1e-3) and rel_fro(gW, rW) <= 1e-6
    assert layer.device_status() == 0
    layer.close()


def test_nearly_overflowing_values_keep_their_products():
    """3.4e38 rounds to infinity in bf16; its products with small values are those of fp32 arithmetic all the same (1e-6)."""
    vbuild.build()
    N, T, d_in, d_out = 2, 40, 72, 64
    X, dY, W = inputs.make_layer(inputs.LayerCase("t", N, T, d_in, d_out, F32, 1.0, 0.5, 0.5, 0.5))
    dY, W, X = dY / dY.abs().max() / 80, W.clone(), X.clone()
    W[5, 7], W[6, 9], X[3, 11] = 3.4e38, -3.4028234e38, 3.3999e38
    layer = vb.Layer(N, T, d_in, d_out, F32)
    dX, dW = layer.dense_bwd(X.cuda(), dY.cuda(), W.cuda())
    rX, rW = np64(dY) @ np64(W), np64(dY).T @ np64(X)
    for got, ref in ((np64(dX), rX), (np64(dW), rW)):
        assert np.isfinite(got).all() and (np.abs(got - ref) <= 1e-6 * np.abs(ref).max(0)).all()
    layer.close()


def same_kind(got, ref):
    """Infinities of the same sign, NaN where NaN, finite where finite."""
    return (np.isnan(got) == np.isnan(ref)).all() and (np.isinf(got) == np.isinf(ref)).all() and \
        (np.sign(got[np.isinf(ref)]) == np.sign(ref[np.isinf(ref)])).all()


@pytest.mark.parametrize("sampled", [True, False])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_infinite_operands(dtype, sampled):
    """Infinities on one or both sides of a product: what IEEE arithmetic gives, inf inf = inf and inf 0 = NaN among it.  At
    ratio 1 every row is kept with scale 1, so the parts of a bf16 layer's rows past the first are 0."""
    vbuild.build()
    N, T, d_in, d_out = 2, 40, 72, 72
    X, dY, W = inputs.make_layer(inputs.LayerCase("t", N, T, d_in, d_out, dtype, 1.0, 0.5, 0.5, 0.5))
    X, dY, W = X.clone(), dY.clone(), W.clone()
    X[50, 3], W[5, 7], dY[20, 8] = float("inf"), float("-inf"), 0.0
    if not sampled:                      # an infinite row norm leaves no probabilities
        dY[3, 5], dY[4, 6], X[4, 9] = float("inf"), float("-inf"), float("inf")
    layer = vb.Layer(N, T, d_in, d_out, dtype)
    args = X.cuda(), dY.cuda(), W.cuda()
    dX, dW = layer.linear_bwd(*args, 1.0, 1.0, 3) if sampled else layer.dense_bwd(*args)
    with np.errstate(invalid="ignore"):
        assert same_kind(np64(dX), np64(dY) @ np64(W)) and same_kind(np64(dW), np64(dY).T @ np64(X))
    layer.close()


def test_layer_whose_parts_do_not_fit_the_device():
    """Rows for 190 GB of parts: the handle is made all the same, with the workspace of the FMA kernels."""
    vbuild.build()
    layer = vb.Layer(512, 2048, 4096, 11008, F32)
    assert layer.workspace_bytes() < 8 * 2**30
    layer.close()
