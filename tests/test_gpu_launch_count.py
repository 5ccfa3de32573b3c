"""profile_read's launch count against the kernel nodes of a captured call:
stages that take several launches (passes of a few ruptures, ranges of K)
count each of them."""
import ctypes
import re

import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402

KERNEL_NODE, RELAXED = 0, 2


def kernel_nodes(call, stream):
    path = re.search(r"\S*libcudart\S*", open("/proc/self/maps").read()).group(0)
    rt = ctypes.CDLL(path)
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), RELAXED) == 0
    try:
        call()
    finally:
        assert rt.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kind, kernels = ctypes.c_int(), 0
    for node in nodes:
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == KERNEL_NODE
    assert rt.cudaGraphDestroy(graph) == 0
    return kernels


@pytest.mark.parametrize("op,prec_g,prec_p,Ns,Ng,B,opts", [
    ("waveforms", "fp32_hilo", "fp32_hilo", 40, 300, 7, {}),  # pairs: two ruptures a launch
    ("waveforms", "fp32", "fp32", 5, 400, 6, {}),  # shortest rows: four a launch
    ("waveforms", "bf16", "bf16", 5, 400, 7, {"engine": "stream"}),  # two a launch
    ("waveforms", "fp32", "fp32", 140, 300, 19, {}),  # three passes
    ("waveforms", "bf16", "bf16", 40, 300, 9, {}),
    ("waveforms", "fp8", "bf16", 40, 300, 40, {"tc_fp8_act": 0}),  # packing: two kernels
    ("adjoint", "fp8", "bf16", 40, 300, 8, {}),  # four ruptures a launch
    ("adjoint", "bf16_hilo", "fp32", 40, 3000, 9, {"tc_adjoint": True})])  # two ranges of K
def test_launches_counted(op, prec_g, prec_p, Ns, Ng, B, opts):
    No, Nt = 6, 32
    ctx = make_context(s2w, compact_box(Ns, Ng, No, seed=Ng), Nt, prec_g=prec_g, prec_p=prec_p, max_batch=B, **opts)
    x = torch.tensor(np.random.default_rng(B).standard_normal((B, Ns if op == "waveforms" else No, Nt)),
                     dtype=torch.float32, device="cuda")
    out = torch.empty((B, No if op == "waveforms" else Ns, Nt), device="cuda")
    stream = torch.cuda.Stream()

    def call():
        if op == "waveforms":
            ctx.waveforms(x, q=out, stream=stream)
        else:
            ctx.adjoint(x, grad=out, stream=stream)
    torch.cuda.synchronize()
    call()  # (loads the kernels)
    ctx.sync()
    before = ctx.profile_read()[1]
    nodes = kernel_nodes(call, stream)
    assert ctx.profile_read()[1] - before == nodes
