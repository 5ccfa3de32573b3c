"""Kernels that are launched before the one ahead of them in the stream has
completed: each waits first thing in its body, calls made back to back on one
stream (inputs written, outputs overwritten by kernels of their own in
between) give the bits of calls made alone, and so does a captured call."""
import glob
import os
import re

import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")

import paper_2608_21763_gb300 as s2w  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.abspath(s2w.__file__)), "csrc")


def test_every_chained_kernel_waits_first():
    src = "".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    direct = set(re.findall(r"launch_next\(\s*(k_\w+)", src))
    through = set(re.findall(r"\b(k_tc_gemm\w*|k_tc_retransform)\b(?=<)", src))  # by pointer, or with clusters
    assert len(direct) > 15 and len(through) > 10
    for name in sorted(direct | through):
        bodies = re.findall(r"__global__[^;{]*?\b%s\([^{;]*\)\s*\{\s*(\w+)" % name, src)
        assert bodies == ["grid_dependency"], (name, bodies)


@pytest.mark.gpu
@pytest.mark.parametrize("prec_g,prec_p,B", [("fp32", "fp32", 1), ("fp32", "fp32", 5), ("fp32_hilo", "fp32_hilo", 2),
                                             ("bf16", "bf16", 9), ("bf16", "bf16", 130), ("bf16_hilo", "fp32", 70),
                                             ("fp8", "bf16", 40), ("fp8", "bf16", 136)])
def test_calls_back_to_back_on_one_stream(prec_g, prec_p, B):
    from test_gpu_parity import compact_box

    Ns, Ng, No, Nt, n = 40, 300, 5, 64, 12
    ctx = make_context(s2w, compact_box(Ns, Ng, No, seed=3), Nt, prec_g=prec_g, prec_p=prec_p, max_batch=B)
    rng = np.random.default_rng(5)
    slips = torch.tensor(rng.standard_normal((n, B, Ns, Nt)).astype(np.float32), device="cuda")
    alone = []
    for i in range(n):
        alone.append(ctx.waveforms(slips[i].contiguous()))
        ctx.sync()
        torch.cuda.synchronize()
    x, q = torch.empty_like(slips[0]), torch.empty_like(alone[0])
    side = torch.cuda.Stream()
    for stream in (torch.cuda.current_stream(), side):
        with torch.cuda.stream(stream):
            got = []
            for i in range(n):
                x.copy_(slips[i])  # the call's input changes between calls ...
                ctx.waveforms(x, q=q)
                got.append(q.clone())
                x.fill_(float("nan"))  # ... and is gone when it returns
                q.fill_(float("nan"))
        torch.cuda.synchronize()
        for i in range(n):
            assert torch.equal(got[i], alone[i]), (i, stream)
    graph = torch.cuda.CUDAGraph()
    x.copy_(slips[0])
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        ctx.waveforms(x, q=q)
    for i in (3, 7):
        x.copy_(slips[i])
        graph.replay()
        assert torch.equal(q, alone[i])
    ctx.sync()
