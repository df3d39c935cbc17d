"""The work this framework is used for, as cases that can be timed one by one.

A training program calls the sampled backward of every linear layer each step, the variance probe every few
hundred steps, the exact backward where it compares or does not sample, and SampleA in front of a LayerNorm.
`listed` names twelve such calls, from the smallest layer to an LLM-sized one; `draw` gives others of the same
ranges.  Layer shapes and value distributions are those of this repository's benchmark (inputs.CASES) or generic.
"""
from __future__ import annotations

import torch

from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import inputs
from paper_2402_17227_b200.stack import LinearStack, StackLayer

DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _case(name, kind, dtype, N, T, d_in, d_out, rho, nu, sigma_A, sigma_B, zero=0.0, M=0, rows=0):
    """kind: sampled | dense | pair | block | probe | layernorm | score.  zero: share of data whose dY is exactly zero.
    M, rows: the probe's batches and the rows of the parameter gradient it samples (0: all of them)."""
    return dict(name=name, kind=kind, dtype=dtype, N=N, T=T, d_in=d_in, d_out=d_out, rho=rho, nu=nu, sigma_A=sigma_A,
                sigma_B=sigma_B, zero=zero, M=M, rows=rows)


def listed():
    return [
        # the smallest layer in use: fp32, 256 rows; launches and latency are all there is
        _case("fp32_small", "sampled", "fp32", 4, 64, 256, 256, 0.5, 0.5, 1.0, 0.5),
        # fine-tuning in full precision: the FFN up-projection of a base-sized transformer in fp32
        _case("fp32_base_ffn_up", "sampled", "fp32", 32, 128, 768, 3072, 0.3, 0.4, 1.5, 1.0),
        # the same layer in bf16: an ordinary fine-tuning step, short kernels
        _case("bert_base_ffn_up", "sampled", "bf16", 32, 128, 768, 3072, 0.3, 0.4, 1.5, 1.0),
        # two linears with a GELU between them, 197 tokens, sparse data handed from one layer to the next
        _case("vit_base_mlp_block", "pair", "bf16", 64, 197, 768, 3072, 0.4, 0.5, 1.2, 0.0),
        # odd sizes: widths that are multiples of 8 only (a classifier of 1000 classes), 150 tokens, 33 data
        _case("ragged_widths", "sampled", "bf16", 33, 150, 776, 1000, 0.5, 0.5, 1.0, 0.5),
        # one transformer block of a large model, four linears in backward order through the stack
        _case("bert_large_block", "block", "bf16", 32, 512, 1024, 4096, 0.5, 0.3, 1.0, 0.5),
        # the largest layer: an LLM's MLP up-projection, 16384 tokens
        _case("llm_mlp_up", "sampled", "bf16", 8, 2048, 4096, 11008, 0.3, 0.3, 0.0, 1.0),
        # the exact backward of the same layer: the comparison, and what a run uses where it does not sample
        _case("llm_mlp_up_dense", "dense", "bf16", 8, 2048, 4096, 11008, 1.0, 1.0, 0.0, 1.0),
        # the probe of that layer on 128 sampled rows of its parameter gradient, once per adaptation period
        _case("llm_probe_128_rows", "probe", "bf16", 8, 2048, 4096, 11008, 0.3, 0.3, 0.0, 1.0, M=2, rows=128),
        # the probe of a base-sized layer on its whole parameter gradient with four Monte-Carlo batches
        _case("bert_base_probe", "probe", "bf16", 32, 128, 768, 3072, 0.3, 0.4, 1.5, 1.0, M=4),
        # SampleA in front of a LayerNorm of a large model
        _case("layernorm_1024", "layernorm", "bf16", 32, 512, 1024, 1024, 0.5, 1.0, 1.0, 0.5),
        # scores, probabilities and kept lists alone (monitoring, or a caller with products of its own)
        _case("bert_large_score", "score", "bf16", 32, 512, 1024, 4096, 0.5, 0.3, 1.0, 0.5),
    ]


def _log_int(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread over its logarithm."""
    v = lo * (hi / lo) ** rng.random()
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["sampled", "sampled", "sampled", "sampled", "dense", "pair", "probe", "layernorm", "score"])
    dtype = "fp32" if kind in ("sampled", "dense", "layernorm", "score") and rng.random() < 0.25 else "bf16"
    # widths: multiples of 64 in most layers, of 8 in the others
    step = 8 if dtype == "fp32" or (kind in ("sampled", "score") and rng.random() < 0.25) else 64
    fma = kind in ("sampled", "dense") and step == 8       # no tensor-core contract there: kept to ordinary sizes
    T = rng.choice([_log_int(rng, 16, 2048), 64, 128, 197, 512])
    N = _log_int(rng, 4, max(4, min(128, (8192 if kind in ("pair", "probe") else 16384) // T)))
    d_in = _log_int(rng, 64, 1536 if fma else 4096, step)
    d_out = _log_int(rng, 64, 4096 if fma else 11008, step)
    if kind in ("pair", "probe"):
        d_in, d_out = min(d_in, 1536), min(d_out, 4096)
    if kind == "layernorm":
        d_in = d_out = max(64, d_in)
    if fma:
        while N * T * d_in * d_out > 4096 * 768 * 3072 and N > 4:
            N -= 1
        while N * T * d_in * d_out > 4096 * 768 * 3072:
            d_out = max(64, d_out // 2 // step * step)
            T = max(16, T // 2)
    rho, nu = rng.choice([1.0, 0.8, 0.5, 0.3, 0.2]), rng.choice([1.0, 0.7, 0.5, 0.3])
    if kind == "dense":
        rho = nu = 1.0
    if kind == "probe":        # at ratio 1 the sampled gradient is the exact one and its variance is rounding noise
        rho, nu = min(rho, 0.8), min(nu, 0.7)
    M = rng.choice([2, 2, 3]) if kind == "probe" else 0
    rows = 64 if kind == "probe" and d_out > 256 and rng.random() < 0.5 else 0
    c = _case("", kind, dtype, N, T, d_in, d_out, rho, nu, rng.choice([0.0, 0.5, 1.0, 1.5]), rng.choice([0.0, 0.5, 1.0]),
              zero=0.0 if kind == "probe" else rng.choice([0.0, 0.0, 0.3]), M=M, rows=rows)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _layer_case(c, seed, d_in, d_out):
    return inputs.LayerCase("case", c["N"], c["T"], d_in, d_out, DTYPES[c["dtype"]], c["sigma_A"], c["sigma_B"], c["rho"],
                            c["nu"], data_seed=seed % 1000003 + 1, zero_fraction=c["zero"])


def _stack_layers(c):
    """(name, d_in, d_out, input is a GELU's output, chained) of a pair or block, in backward order."""
    d, ff = c["d_in"], c["d_out"]
    mlp = [("mlp_down", ff, d, True, False), ("mlp_up", d, ff, False, True)]
    return mlp if c["kind"] == "pair" else mlp + [("attn_out", d, d, False, False), ("qkv", d, 3 * d, False, False)]


def prepare(case, seed):
    """Inputs, output buffers and the handle that a training program keeps for this layer shape."""
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    N, T, d_in, d_out, dt = c["N"], c["T"], c["d_in"], c["d_out"], DTYPES[c["dtype"]]
    s = dict(kind=c["kind"], rho=c["rho"], nu=c["nu"], seed=seed % 65521 + 1)
    if c["kind"] in ("pair", "block"):
        layers = []
        for i, (name, di, do, gelu, chained) in enumerate(_stack_layers(c)):
            lc = _layer_case(c, seed + i, di, do)
            X, dY, W = inputs.make_layer(lc, device=dev)
            H = [inputs.make_preactivation(lc, device=dev)] if gelu else None
            layers.append(StackLayer(name, di, do, W, [X], [] if chained else [dY], H=H, chained=chained))
        s["stack"] = LinearStack(layers, N, T, dt, overlap_layers=True)
        s["rhos"], s["nus"] = [c["rho"]] * len(layers), [c["nu"]] * len(layers)
        return s
    lc = _layer_case(c, seed, d_in, d_out)
    s["layer"] = vb.Layer(N, T, d_in, d_out, dt)
    if c["kind"] == "probe":
        if c["rows"]:
            s["layer"].set_probe_subsample(c["rows"], seed=1)
        batches = [inputs.make_layer(lc, batch=b, device=dev) for b in range(c["M"])]
        s["Xs"], s["dYs"], s["W"] = [b[0] for b in batches], [b[1] for b in batches], batches[0][2]
        return s
    s["X"], s["dY"], s["W"] = inputs.make_layer(lc, device=dev)
    if c["kind"] == "layernorm":
        g = torch.Generator(dev).manual_seed(seed % 1000003 + 5)
        s["gamma"] = (1.0 + 0.2 * torch.randn(d_in, generator=g, device=dev)).to(dt)
    if c["kind"] in ("sampled", "dense", "layernorm"):
        s["dX"] = torch.empty(N * T, d_in, dtype=dt, device=dev)
    if c["kind"] in ("sampled", "dense"):
        s["dW"] = torch.empty(d_out, d_in, dtype=torch.float32, device=dev)
    return s


def run(s):
    kind = s["kind"]
    if kind == "sampled":
        s["layer"].linear_bwd_plain(s["X"], s["dY"], s["W"], s["rho"], s["nu"], s["seed"], s["dX"], s["dW"])
        return [s["dX"], s["dW"]]
    if kind == "dense":
        return list(s["layer"].dense_bwd(s["X"], s["dY"], s["W"], dX=s["dX"], dW=s["dW"]))
    if kind in ("pair", "block"):
        s["stack"].backward(s["rhos"], s["nus"], s["seed"])
        # the last layer's dX, and the dX handed down to the chained layer
        return [L.dW for L in s["stack"].layers] + [s["stack"].layers[0].dX, s["stack"].layers[-1].dX]
    if kind == "probe":
        out = s["layer"].variance_probe(s["Xs"], s["dYs"], s["W"], s["rho"], s["nu"], 0.8, s["seed"])
        return dict(zip(("V_s", "V_act", "V_w", "p_lo", "p_hi"), out.unbind()))
    if kind == "layernorm":
        return list(s["layer"].layernorm_bwd(s["X"], s["gamma"], s["dY"], s["rho"], s["seed"], dX=s["dX"]))
    r = s["layer"].score(s["X"], s["dY"], s["rho"], s["nu"], s["seed"])
    kept = torch.zeros(r.q.numel(), dtype=torch.bool, device=r.q.device)      # the kept rows, as a mask of fixed length
    kept[r.idxW] = True
    return [r.g, r.p, r.w, r.q, kept]


# --------------------------------------------------------------------------------- work and tolerance
def _linear_work(R, d_in, d_out, b, rho, nu, chained, gelu, dense=False):
    """One backward: dY is read whole for its norms (not when the layer above hands them down; then its kept rows),
    X on the rows of kept data, W, and with a GELU its pre-activation on those rows; dX and dW are written."""
    kept = rho * R
    dy_rows = R if dense or not chained else kept
    by = (dy_rows * d_out + kept * d_in + d_out * d_in + R * d_in + (kept * d_in if gelu else 0)) * b + d_out * d_in * 4
    return by, 2.0 * kept * d_in * d_out * (1.0 + nu)


def work(case):
    c = case
    R, d_in, d_out, b = c["N"] * c["T"], c["d_in"], c["d_out"], 4 if c["dtype"] == "fp32" else 2
    rho, nu, kind = c["rho"], c["nu"], c["kind"]
    if kind in ("sampled", "dense"):
        by, fl = _linear_work(R, d_in, d_out, b, rho, nu, False, False, kind == "dense")
    elif kind in ("pair", "block"):
        by = fl = 0.0
        for _, di, do, gelu, chained in _stack_layers(c):
            y, f = _linear_work(R, di, do, b, rho, nu, chained, gelu)
            by, fl = by + y, fl + f
    elif kind == "probe":
        # per batch the exact gradient and M sampled ones, on all or on the sampled rows of the parameter gradient
        M, rows = c["M"], c["rows"] or d_out
        by = M * R * (d_in + d_out) * b + 20.0
        fl = M * 2.0 * R * d_in * rows * (1.0 + M * rho)
    elif kind == "layernorm":
        by = (R * d_in + rho * R * d_in + R * d_in + d_in) * b + 2 * d_in * 4
        fl = R * d_in * (2.0 + 20.0 * rho)
    else:
        by = R * d_out * b + rho * R * d_in * b + R * 12.0
        fl = 2.0 * R * (d_out + rho * d_in)
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    """Four times what was measured: fp32 results against their sums in 64 bits 1e-6 (up to 3072 terms; more terms are
    drawn), 1.7e-3 for bf16 (dX is rounded to bf16 once, and so are the rescaled rows of dY that enter the dW product;
    another correct kernel may round elsewhere), 3e-5 for the probe's scalars under another order of its sums.  A row
    whose uniform lies within rounding of its keep probability may fall on either side."""
    if case["kind"] == "score":
        return {"rel": 1e-5, "differ": 1e-3}
    if case["kind"] == "probe":
        return {"rel": 2e-4}
    return {"rel": 1e-5 if case["dtype"] == "fp32" else 7e-3}
