"""Several ruptures per pass of the transposed streaming kernel (the adjoint):
a batch must give, bit for bit, what its ruptures give one at a time, and the
gradient must satisfy the adjoint identity <q(s), r> = <s, grad(r)> with the
forward map, at the edges of the row chunks (512), stages, column groups and
passes (8 ruptures)."""
import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


@pytest.mark.parametrize("prec", ["fp32", "bf16", "bf16_hilo", "fp8"])
@pytest.mark.parametrize("Ns,Ng,No,Nt,B", [(1, 37, 1, 32, 2), (260, 513, 64, 32, 9), (1024, 512, 3, 64, 8),
                                           (501, 1100, 33, 32, 5), (9, 640, 120, 32, 17), (968, 100, 2, 256, 3)])
def test_adjoint_batch(prec, Ns, Ng, No, Nt, B):
    geom = compact_box(Ns, Ng, No, seed=Ns + Ng)
    rng = np.random.default_rng(B)
    slip = torch.tensor(rng.standard_normal((B, Ns, Nt)), dtype=torch.float32, device="cuda")
    r = torch.tensor(rng.standard_normal((B, No, Nt)), dtype=torch.float32, device="cuda")
    ctx = make_context(s2w, geom, Nt, prec_g=prec, prec_p="bf16" if prec in ("bf16", "fp8") else "fp32",
                       max_batch=B, chunk=1024, engine="stream")
    g = ctx.adjoint(r)
    for b in range(B):
        assert torch.equal(ctx.adjoint(r[b:b + 1].contiguous())[0], g[b]), b
    q = ctx.waveforms(slip)
    lhs = (q.double() * r.double()).sum((1, 2))
    rhs = (slip.double() * g.double()).sum((1, 2))
    scale = q.double().flatten(1).norm(dim=1) * r.double().flatten(1).norm(dim=1)
    scale = scale + slip.double().flatten(1).norm(dim=1) * g.double().flatten(1).norm(dim=1)
    # both maps apply the same stored operators; the forward FP8 kernel also
    # rounds its vector to FP16 (2^-11 per entry), the rest is FP32 rounding
    # on the scale of the 2 Nt window
    tol = 1e-3 if prec == "fp8" else 1e-5
    assert torch.all((lhs - rhs).abs() <= tol * scale)
    ctx.sync()
