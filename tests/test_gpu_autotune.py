"""What the autotuner's choices rest on."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402


def random_context(Ns, Ng, No, Nt, **kw):
    ctx = s2w.Context(Ns, Ng, No, Nt, **kw)
    gen = torch.Generator(device="cuda").manual_seed(Ns)
    ctx.load_greens(0, torch.randn(Ng, Ns, Nt, device="cuda", generator=gen))
    ctx.load_adjoint(0, torch.randn(No, Ng, Nt, device="cuda", generator=gen))
    return ctx


def test_threshold_compares_the_engines_on_the_same_batch():
    """Four ruptures of this workload take the streaming kernels (one pass of
    the operators) 0.107 ms and the tensor engine 0.134, sixteen 0.33 and
    0.150: the tuned threshold lies between."""
    ctx = random_context(200, 2000, 16, 128, prec_g="bf16_hilo", prec_p="fp32", max_batch=32)
    t = ctx.autotune(32)
    print(t)
    assert 4 < t["tc_min_batch"] <= 16
