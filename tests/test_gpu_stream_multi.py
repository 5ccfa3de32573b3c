"""Several ruptures per pass of the streaming kernels: a batch must give, bit
for bit, what its ruptures give one at a time (the single-rupture kernels,
which the parity tests hold to the oracle), at the edges of the row tiles (64
rows), of the row lengths (64 chunks of 16 bytes), of the passes (8 ruptures)
and of the short and long row kernels."""
import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


# rows of up to 16 chunks (Ns = 32 FP32, 64 BF16) stay on lane groups, longer
# ones go to the tiled kernel; one rupture's short rows end at 64 chunks (Ns =
# 128, 256); stage 2's rows are the grid segments
@pytest.mark.parametrize("prec", ["fp32", "bf16", "bf16_hilo", "fp8"])
@pytest.mark.parametrize("Ns,Ng,No,Nt,B", [(129, 63, 1, 32, 2), (128, 64, 9, 32, 9), (257, 65, 64, 32, 5),
                                           (1024, 130, 65, 64, 8), (300, 1100, 3, 32, 17), (5, 400, 120, 32, 6),
                                           (264, 257, 8, 256, 3), (40, 200, 3, 32, 8), (100, 90, 70, 64, 6), (70, 70, 9, 32, 4)])
def test_batch_equals_single_ruptures_bitwise(prec, Ns, Ng, No, Nt, B):
    geom = compact_box(Ns, Ng, No, seed=Ns + Ng)
    slip = torch.tensor(np.random.default_rng(B).standard_normal((B, Ns, Nt)), dtype=torch.float32, device="cuda")
    ctx = make_context(s2w, geom, Nt, prec_g=prec, prec_p="bf16" if prec in ("bf16", "fp8") else "fp32",
                       max_batch=B, chunk=1024, engine="stream")
    m = torch.empty((B, Ng, Nt), device="cuda")
    q = ctx.waveforms(slip, seafloor=m)
    for b in range(B):
        m1 = torch.empty((1, Ng, Nt), device="cuda")
        q1 = ctx.waveforms(slip[b:b + 1].contiguous(), seafloor=m1)
        assert torch.equal(q1[0], q[b]) and torch.equal(m1[0], m[b]), b
    # the seafloor field in host memory takes one rupture at a time
    qh, mh = np.empty((B, No, Nt), np.float32), np.empty((B, Ng, Nt), np.float32)
    ctx.waveforms(slip.cpu().numpy(), q=qh, seafloor=mh)
    assert np.array_equal(qh, q.cpu().numpy()) and np.array_equal(mh, m.cpu().numpy())
    ctx.sync()


@pytest.mark.parametrize("B", [2, 7])
def test_single_pass_batch_equals_single_ruptures_bitwise(B):
    Ns, Ng, No, Nt = 140, 300, 5, 32
    geom = compact_box(Ns, Ng, No, seed=4)
    slip = torch.tensor(np.random.default_rng(B).standard_normal((B, Ns, Nt)), dtype=torch.float32, device="cuda")
    ctx = make_context(s2w, geom, Nt, max_batch=B, engine="stream", single_pass=True)
    q = ctx.waveforms(slip)
    for b in range(B):
        assert torch.equal(ctx.waveforms(slip[b:b + 1].contiguous())[0], q[b]), b
    ctx.sync()
