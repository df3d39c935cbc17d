"""Helpers of the GPU parity tests: tensor conversion and error norms."""
import numpy as np
import torch

from oracle import vcas_oracle as o


def f32(x: float) -> float:
    """The value a float takes when it crosses the C ABI as `float`."""
    return float(np.float32(x))


def np64(t: torch.Tensor) -> np.ndarray:
    """Exact float64 copy of a stored tensor (bf16 and fp32 values are representable)."""
    return t.detach().float().cpu().numpy().astype(np.float64)


def rel_fro(a, b) -> float:
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    nb = np.linalg.norm(b)
    return float(np.linalg.norm(a - b) / nb) if nb > 0 else float(np.linalg.norm(a))


def tol_for(dtype) -> float:
    """Relative Frobenius tolerance of dX and dW: 1e-5 for the fp32 path, 2e-2 for bf16 inputs
    with fp32 accumulation (bf16 outputs carry 2^-9 rounding per element, about 2e-3 in norm)."""
    return 1e-5 if dtype == torch.float32 else 2e-2


def v_act_of_rounded_rows(layer, batches, rho, seed, param_rows):
    """V_act of the probe in float64 on the rows the library multiplies: those of kept data rescaled by 1/p, at the library's own
    p, and rounded to bf16.  batches: (X, dY, W) on the host."""
    N, T, M = layer.N, layer.T, len(batches)
    rows = slice(None) if param_rows is None else param_rows
    total = 0.0
    for i, (X, dY, _) in enumerate(batches):
        p = layer.score(X.cuda(), dY.cuda(), rho, 0.5, 1).p.cpu()
        keep = [o.bernoulli_keep(p.numpy(), o.probe_seed(seed, i, j, M), 0) for j in range(M)]
        sc = (1.0 / p).repeat_interleave(T)[:, None]
        E = np64((dY.float() * sc).to(torch.bfloat16))[:, rows]      # 1/p and the product rounded to fp32, then to bf16
        G_s = np64(dY)[:, rows].T @ np64(X)
        for k in keep:
            kr = np.repeat(k, T)
            total += float((((E[kr].T @ np64(X)[kr]) - G_s) ** 2).sum())
    d_out = batches[0][1].shape[1]
    return total / (M * M) * (1.0 if param_rows is None else d_out / len(param_rows))
