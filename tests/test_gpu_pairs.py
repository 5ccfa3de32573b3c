"""The FP32-pair kernels at the edges of their shapes: rows of 4, 8, 9, 16, 17,
31, 32, 33 and 512 chunks (lane groups, whole warps, slabs), row tiles cut by
the grid and the observations, every transform length, one, two and three
ruptures per call.  The FP64 oracle, at the precision's own bar (1e-5 plain
relative L2; FP32 rounding of the waveforms alone is 3e-8, and 2e-7 is
asserted where the kept head is at least a tenth of its FFT window); a batch
gives the same bits as its ruptures alone."""
import numpy as np
import pytest

import oracle
from helpers import make_context, window_norms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2608_21763_gb300 as s2w  # noqa: E402
from test_gpu_parity import compact_box  # noqa: E402


@pytest.mark.parametrize("Ns,Ng,No,Nt", [(7, 37, 1, 32), (16, 300, 5, 64), (18, 129, 33, 32), (32, 65, 64, 128),
                                         (34, 1025, 3, 32), (62, 70, 2, 256), (64, 257, 9, 32), (66, 40, 65, 64),
                                         (1024, 30, 2, 512)])
def test_pair_contractions_and_transforms(Ns, Ng, No, Nt):
    B = 3
    geom = compact_box(Ns, Ng, No, seed=Ns)
    slip = np.random.default_rng(Ns).standard_normal((B, Ns, Nt)).astype(np.float32)
    slip[:, :, Nt // 2:] = 0
    ctx = make_context(s2w, geom, Nt, prec_g="fp32_hilo", prec_p="fp32_hilo", max_batch=B)
    x = torch.tensor(slip, device="cuda")
    m = torch.empty((B, Ng, Nt), device="cuda")
    q = ctx.waveforms(x, seafloor=m)
    for b in range(B):
        assert torch.equal(ctx.waveforms(x[b:b + 1].contiguous())[0], q[b]), b
    assert torch.equal(ctx.waveforms(x[:2].contiguous()), q[:2])
    ctx.sync()
    # the operators as the library was given them
    G = geom.greens_rows(0, Ng, Nt, np.float32).astype(np.float64)
    P = geom.adjoint_cols(0, Ng, Nt, np.float32).astype(np.float64)
    q_ref, m_ref = oracle.waveforms(G, P, slip.astype(np.float64), return_seafloor=True)
    _, kappa = window_norms(G, P, slip.astype(np.float64))
    err = np.linalg.norm((q.cpu().numpy() - q_ref).reshape(B, -1), axis=1) / np.linalg.norm(q_ref.reshape(B, -1), axis=1)
    assert np.all(err <= np.where(kappa <= 10, 2e-7, 1e-5)), (err, kappa)
    assert np.linalg.norm(m.cpu().numpy() - m_ref) <= 2e-7 * np.linalg.norm(m_ref)
