"""How exactly the streaming kernels sum a long row.  Responses and slip that
act at the first sample alone have flat, real spectra: both transforms are
exact on them, and the seafloor field's first sample is the FP32 dot product
of a row with the slip as the kernel forms it.  Its rounding must be that of
two accumulations per lane, each over half of the lane's products (emulated
here), which is what the error figures of the stream engine rest on; one
accumulation per lane rounds 1.2 times as much at these lengths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2608_21763_gb300 as s2w  # noqa: E402


def two_accumulations(g, x, C):
    """FP32 dot products of rows g [n][cols] with x [cols]: 16-byte chunks of C
    entries dealt to 32 lanes, even and odd entries of a lane apart, the lanes
    added over xor 16, 8, .. 1."""
    n, cols = g.shape
    slabs = -(-cols // (32 * C))
    pad = slabs * 32 * C - cols
    g = np.pad(g, ((0, 0), (0, pad))).reshape(n, slabs, 32, C)
    x = np.pad(x, (0, pad)).reshape(slabs, 32, C)
    acc = np.zeros((2, n, 32), np.float32)
    for t in range(slabs):
        for q in range(C):
            p = g[:, t, :, q].astype(np.float64) * x[t, :, q].astype(np.float64)  # exact; one rounding below: an FMA
            acc[q % 2] = (acc[q % 2].astype(np.float64) + p).astype(np.float32)
    v = acc[0] + acc[1]
    for o in (16, 8, 4, 2, 1):
        v = v + v[:, np.arange(32) ^ o]
    return v[:, 0]


# Of two samples of n errors each the ratio of their root mean squares is 1 +-
# n^-1/2: four of that at n = 4,096 gives the bound.
BOUND = 1 + 4 * 4096 ** -0.5


@pytest.mark.gpu
@pytest.mark.parametrize("prec,Ns", [("fp32", 1024), ("fp32", 968), ("bf16", 1024), ("bf16_hilo", 1024)])
@pytest.mark.parametrize("per_call", [8, 6, 4, 2, 1])
def test_long_rows_round_like_two_accumulations(prec, Ns, per_call):
    B, Ng, No, Nt = 8, 512, 1, 32
    rng = np.random.default_rng(Ns)
    a = torch.tensor(rng.standard_normal((Ng, Ns)), dtype=torch.float32).bfloat16().float()  # exact in every storage
    s = torch.tensor(rng.standard_normal((B, Ns)), dtype=torch.float32)
    G, slip = torch.zeros((Ng, Ns, Nt), device="cuda"), torch.zeros((B, Ns, Nt), device="cuda")
    G[:, :, 0], slip[:, :, 0] = a.cuda(), s.cuda()
    ctx = s2w.Context(Ns, Ng, No, Nt, prec_g=prec, prec_p="fp32", max_batch=B, engine="stream")
    ctx.load_greens(0, G)
    ctx.load_adjoint(0, torch.ones((No, Ng, Nt), device="cuda"))
    m = torch.empty((B, Ng, Nt), device="cuda")
    for b in range(0, B, per_call):
        ctx.waveforms(slip[b:b + per_call], seafloor=m[b:b + per_call])
    ctx.sync()
    m, a, s = m.cpu().numpy(), a.numpy(), s.numpy()
    assert not m[:, :, 1:].any()
    exact = s.astype(np.float64) @ a.T.astype(np.float64)
    ref = np.stack([two_accumulations(a, s[b], 2 if prec == "fp32" else 4) for b in range(B)])
    rms = np.sqrt(np.mean((m[:, :, 0] - exact) ** 2)) / np.sqrt(np.mean((ref - exact) ** 2))
    print(f"{prec} {Ns}, {per_call} per call: rounding against two accumulations {rms:.3f}")
    assert rms <= BOUND
