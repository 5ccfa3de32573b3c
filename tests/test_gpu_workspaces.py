"""Device memory of a context: the streaming kernels' workspaces are kept for
as many ruptures as share a pass of the operators on that context, not more."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402

Ns, Ng, No, Nt = 256, 60000, 2, 32
SET = 8 * (Nt + 1) * Ng  # seafloor (or velocity) spectra of one rupture
GPART = 8 * (Nt + 1) * -(-Ng // 512) * Ns  # adjoint partials of one rupture
SLACK = 24 << 20  # allocation granules, and what else grows with the batch (slip, residuals, partials)


def held(max_batch, **kw):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = s2w.Context(Ns, Ng, No, Nt, max_batch=max_batch, **kw)
    got = before - torch.cuda.mem_get_info()[0]
    del ctx
    return got


# sets: of seafloor, velocity spectra and adjoint partials per rupture past the
# first that the context may keep; tc: bytes per grid point, bin and rupture
# of the tensor engine's own operands (BF16 seafloor and velocity spectra)
@pytest.mark.parametrize("kw,sets,parts,tc", [
    (dict(prec_g="fp32", prec_p="fp32"), 7, 7, 0),
    (dict(prec_g="fp32_hilo", prec_p="fp32_hilo"), 2, 0, 0),  # one more rupture, hi and lo
    (dict(prec_g="bf16", prec_p="bf16", engine="tensor"), 0, 0, 8),
    (dict(prec_g="bf16", prec_p="bf16", engine="stream"), 7, 7, 0),
    (dict(prec_g="fp8", prec_p="bf16", engine="stream"), 3, 3, 0),
    (dict(prec_g="fp8", prec_p="bf16", engine="tensor"), 0, 0, 8)])
def test_workspaces_fit_the_engine(kw, sets, parts, tc):
    held(1, **kw)  # (the first context of a process also loads the library's code)
    more = held(8, **kw) - held(1, **kw)
    assert more <= sets * 2 * SET + parts * GPART + 7 * tc * (Nt + 1) * Ng + SLACK, more
