"""Kernels that read ahead of their wait for the kernel before them (the two that emit kept rows).  What that rests on stands in
the sources: the kernel in front waits before it lets them start, and they read past L1.  On the GPU: calls that follow one another
on a handle, with other inputs every time, give bit for bit what handles of their own give."""
import os
import re

import pytest
import torch

from paper_2402_17227_b200 import binding as vb
from paper_2402_17227_b200 import build as vbuild
from paper_2402_17227_b200 import inputs


def body(src, name):
    """The text of the function `name`, from its name to the end of its braces."""
    at = re.search(r"\b%s\([^;]*?\)\s*\{" % name, src)
    depth, i = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[at.start():i]


def test_order_and_loads_in_the_sources():
    with open(os.path.join(vbuild.CSRC, "sampler.cu")) as f:
        src = re.sub(r"//.*", "", f.read())
    for name in ("sample_w_small_kernel", "sample_w_kernel"):
        k = body(src, name)
        assert 0 < k.index("pdl_wait()") < k.index("pdl_trigger()"), name
    memory = re.compile(r"(?<!__ldcg\()(?<!read\()P\.(idxA|dropA|wc|uc|scaleA|counts|w|q|fix|chunk_off)\b(?! !=)")
    k = body(src, "chunk_in")
    assert not memory.findall(k) and "return AHEAD ? __ldcg(p) : *p;" in k
    for name in ("emit_rows_kernel", "emit_pack_kernel"):
        before = body(src, name).split("pdl_wait()")[0]
        assert not memory.findall(before) and "chunk_in<true>(" in before and "chunk_in<false>(" not in before, name


@pytest.mark.gpu
@pytest.mark.parametrize("N,T,d_in,d_out,dtype", [(4, 64, 64, 64, torch.bfloat16), (40, 100, 128, 72, torch.bfloat16),
                                                  (9, 33, 64, 200, torch.float32), (37, 500, 64, 64, torch.bfloat16)])
def test_other_inputs_every_call(N, T, d_in, d_out, dtype):
    vbuild.build()
    sets = []
    for i, rho in enumerate((0.2, 0.9, 0.5)):
        case = inputs.LayerCase("ra", N, T, d_in, d_out, dtype, 1.0, 0.5, rho, 0.5, data_seed=11 + i)
        X, dY, W = (t.cuda() for t in inputs.make_layer(case))
        alone = vb.Layer(N, T, d_in, d_out, dtype)
        out = alone.linear_bwd(X, dY, W, rho, 0.5, i)
        s = alone.score(X, dY, rho, 0.5, i)
        sets.append((X, dY, W, rho, i, out, s))
        assert alone.device_status() == 0
        alone.close()
    layer, got = vb.Layer(N, T, d_in, d_out, dtype), []
    for k in range(12):
        X, dY, W, rho, i, _, _ = sets[k * 5 % 3]
        got.append((k * 5 % 3, layer.linear_bwd(X, dY, W, rho, 0.5, i)))
    for j, out in got:
        assert torch.equal(out[0], sets[j][5][0]) and torch.equal(out[1], sets[j][5][1])
    for k in range(6):
        X, dY, W, rho, i, _, s = sets[k * 2 % 3]
        r = layer.score(X, dY, rho, 0.5, i)
        assert torch.equal(r.q, s.q) and torch.equal(r.w, s.w) and torch.equal(r.idxW, s.idxW) and r.cntA == s.cntA
    assert layer.device_status() == 0
    layer.close()
