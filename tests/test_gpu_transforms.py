"""The row transforms (zero-padded real FFT, truncated inverse) at the edges of
their launches: one row, fewer and more rows than a CTA's warps, more rows
than the persistent grid has warps, and buffers that are only 4-byte aligned;
and the transposed form (slip spectra) through a context whose row count
crosses its tile shapes.  Reference: torch's FP64 FFT.  Bound: an FP32 FFT of
length 2 Nt errs by about 2^-24 sqrt(log2(2 Nt)) of the signal per stage set,
under 4e-7 relative in L2 at 1,024 points; 1e-6 is asserted."""
import numpy as np
import pytest

from helpers import make_context

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


def shifted(shape, dtype, off):
    n = int(np.prod(shape))
    return torch.empty(n + off, dtype=dtype, device="cuda")[off:].view(shape)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("rows", [1, 7, 9, 4000])
@pytest.mark.parametrize("Nt", [32, 64, 128, 256, 512])
def test_row_transforms(Nt, rows, off):
    ctx = s2w.Context(4, 8, 2, Nt)
    x = shifted((rows, Nt), torch.float32, off)
    x.copy_(torch.randn(rows, Nt, generator=torch.Generator(device="cuda").manual_seed(rows), device="cuda"))
    X = ctx.rfft(x)
    ref = torch.fft.rfft(x.double(), n=2 * Nt)
    assert float((X.to(torch.complex128) - ref).norm() / ref.norm()) <= 1e-6
    y = ctx.irfft(X, x=shifted((rows, Nt), torch.float32, off))
    assert float((y.double() - x.double()).norm() / x.double().norm()) <= 1e-6
    ctx.sync()


@pytest.mark.parametrize("Nt", [32, 128, 256, 512])
@pytest.mark.parametrize("Ns,B", [(3, 1), (31, 2), (33, 160)])
def test_transposed_rows_do_not_depend_on_the_tile(Nt, Ns, B):
    """Few rows go in tiles of 8, many in tiles of 16 or 32: the waveforms of a
    rupture are the same bits in a batch and alone, for even and odd row
    counts and for active lengths that end inside a sample pair."""
    geom = compact_box(Ns, 40, 2, seed=Ns)
    slip = torch.tensor(np.random.default_rng(Ns).standard_normal((B, Ns, Nt)), dtype=torch.float32, device="cuda")
    ctx = make_context(s2w, geom, Nt, max_batch=B, engine="stream")
    lens = [(7 * b + 1) % (Nt + 1) for b in range(B)]
    q = ctx.waveforms_active(slip, lens)
    for b in {0, B // 2, B - 1}:
        z = slip[b:b + 1].clone()
        z[:, :, lens[b]:] = 0
        assert torch.equal(ctx.waveforms(z)[0], q[b]), b
    ctx.sync()
