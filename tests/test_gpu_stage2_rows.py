"""Stage 2 of the tensor engine with fewer ruptures than a tile's 128 rows:
stages that keep only the live rows (8 to 120 of them, rings from 3 to 24
stages deep, K blocks past a lap of the ring) give the bits of the same
ruptures in a batch of 128, where every row is live."""
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


@pytest.mark.parametrize("No", [1, 16, 17, 63, 128])
@pytest.mark.parametrize("Ng", [37, 2003])
def test_live_rows_only(No, Ng):
    Ns, Nt, full = 9, 32, 128
    ctx = make_context(s2w, compact_box(Ns, Ng, No, seed=No), Nt, prec_g="bf16", prec_p="bf16", max_batch=full,
                       engine="tensor")
    x = torch.randn(full, Ns, Nt, generator=torch.Generator(device="cuda").manual_seed(No), device="cuda")
    q = ctx.waveforms(x)
    assert torch.isfinite(q).all() and float(q.abs().max()) > 0
    for B in (1, 7, 8, 9, 33, 64, 119, 120, 121, 127):
        assert torch.equal(ctx.waveforms(x[:B].contiguous()), q[:B]), B
        assert torch.equal(ctx.waveforms(x[full - B:].contiguous()), q[full - B:]), B
    ctx.sync()
