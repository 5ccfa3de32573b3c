"""A residual that is not finite (a gap in the targets) spoils its own gradient
and nothing else: later calls on the context give the bits of a context that
never saw it."""
import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


# grids that end inside a padded segment, on an odd and an even column, for
# rows on one and on several groups of threads
@pytest.mark.parametrize("prec,Ns,Ng,Nt", [("fp32", 40, 301, 32), ("fp32", 33, 1100, 32), ("fp32", 9, 1021, 32),
                                           ("bf16", 40, 2050, 64), ("bf16_hilo", 24, 77, 32), ("fp8", 40, 999, 32)])
def test_forward_after_an_adjoint_that_is_not_finite(prec, Ns, Ng, Nt):
    No, B = 6, 8
    geom = compact_box(Ns, Ng, No, seed=Ng)
    rng = np.random.default_rng(Ng)
    slip = torch.tensor(rng.standard_normal((B, Ns, Nt)), dtype=torch.float32, device="cuda")
    r = torch.tensor(rng.standard_normal((B, No, Nt)), dtype=torch.float32, device="cuda")

    def context():
        return make_context(s2w, geom, Nt, prec_g=prec, prec_p="bf16" if prec in ("bf16", "fp8") else "fp32",
                            max_batch=B, engine="stream")
    fresh, ctx = context(), context()
    q, g = fresh.waveforms(slip), fresh.adjoint(r)
    for bad in (float("nan"), float("inf")):
        gap = r.clone()
        gap[B - 1, No - 1, Nt // 2] = bad
        g_bad = ctx.adjoint(gap)
        assert torch.equal(g_bad[:B - 1], g[:B - 1]) and not torch.isfinite(g_bad[B - 1]).all()
        ctx.adjoint(r[:1].contiguous())
        assert torch.equal(ctx.waveforms(slip), q)
        assert torch.equal(ctx.adjoint(r), g)
    ctx.sync()
