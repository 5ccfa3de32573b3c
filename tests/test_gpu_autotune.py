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


def test_cache_entries_of_earlier_kernels_are_timed_again(tmp_path):
    """An entry without the revision of the kernels that it was timed on is
    not applied; it stays in the file, and the new entry is."""
    import re

    cache = tmp_path / "tune.txt"
    kw = dict(prec_g="bf16", prec_p="bf16", max_batch=8, tune_cache=str(cache))
    assert not random_context(24, 700, 6, 64, **kw).autotune(8)["from_cache"]
    line = cache.read_text()
    earlier = re.sub(r",rev=\d+", "", line)
    cache.write_text(earlier)
    ctx = random_context(24, 700, 6, 64, **kw)
    assert not ctx.autotune(8)["from_cache"]
    assert earlier in cache.read_text() and cache.read_text().count("\n") == 2
    assert ctx.autotune(8)["from_cache"]
