"""The call without allocation: problems that fit its scratch."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402


def test_pairs_with_many_observations_fit():
    """A small grid with many observations on FP32 pairs: 7 MB of spectra and
    partials (of one segment each), the same bits as the allocating call."""
    Ns, Ng, No, Nt = 8, 1024, 9000, 32
    gen = torch.Generator(device="cuda").manual_seed(1)
    ctx = s2w.Context(Ns, Ng, No, Nt, prec_g="fp32_hilo", prec_p="fp32_hilo")
    ctx.load_greens(0, torch.randn(Ng, Ns, Nt, device="cuda", generator=gen))
    for g0 in range(0, Ng, 256):
        ctx.load_adjoint(g0, torch.randn(No, 256, Nt, device="cuda", generator=gen))
    slip = torch.randn(1, Ns, Nt, device="cuda", generator=gen)
    q, ref = torch.full((No, Nt), float("nan"), device="cuda"), ctx.waveforms(slip)[0]
    stream = torch.cuda.current_stream().cuda_stream
    status = s2w.lib().s2w_waveforms_noalloc(ctx._h, slip.data_ptr(), q.data_ptr(), stream)
    assert status == 0, s2w.lib().s2w_last_error(ctx._h)
    ctx.sync()
    assert torch.equal(q, ref)
