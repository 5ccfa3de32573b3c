"""The workloads that the library's speed is judged by.

Each case is one call of a public entry point on a context whose operators
are loaded (the spectra are computed once and kept; loading is the setup of a
user's program).  Operators, ruptures and targets are made on the GPU from
the seed alone: Ricker responses delayed by travel time between a dipping
fault plane, the seafloor grid over it and the observations, and ruptures
that spread from a hypocentre with triangular slip-rate functions, the same
kind of inputs as the repository's generator on sizes of its named workloads
(963 subfaults, 64 observations, 256 steps and the paper's per-GPU shapes).
Grids are cut down where three contexts would not fit the card.

``op``: waveforms; active (uneven durations); seafloor (the motion field is
returned too); gradient (misfit gradient in one call); autograd (the
differentiable misfit, forward and backward); transforms (the zero-padded
real FFT of rows and its truncated inverse).
"""
import math

import numpy as np
import torch

import paper_2608_21763_gb300 as s2w
from paper_2608_21763_gb300 import autograd

DEV = "cuda:0"
GREEN_KMS, ADJ_KMS, DECAY_KM, F0_HZ, RUPTURE_KMS = 3.5, 0.2, 50.0, 0.1, 2.8


def _case(name, op, prec_g, prec_p, Ns, Ng, No, Nt, B, tc_adjoint=False):
    return {"name": name, "op": op, "prec_g": prec_g, "prec_p": prec_p, "Ns": Ns, "Ng": Ng, "No": No, "Nt": Nt,
            "B": B, "tc_adjoint": tc_adjoint}


def listed():
    return [
        # two ruptures of the tiny workload on the accurate (FP32 pair) path: latency and launches
        _case("tiny_pairs_b2", "waveforms", "fp32_hilo", "fp32_hilo", 16, 1024, 4, 32, 2),
        # the plain workload: one rupture, default precision, operators of the paper's shape
        _case("plain_fp32_b1", "waveforms", "fp32", "fp32", 963, 20000, 64, 256, 1),
        # a small ensemble at the default precision on the paper's weak-scaling shape
        _case("weak_fp32_b8", "waveforms", "fp32", "fp32", 480, 37758, 32, 256, 8),
        # one rupture on FP32 pairs, for records whose energy arrives late
        _case("csz_pairs_b1", "waveforms", "fp32_hilo", "fp32_hilo", 963, 6000, 64, 256, 1),
        # a handful of ruptures on BF16 operators: the low end of the tensor engine
        _case("bf16_b8", "waveforms", "bf16", "bf16", 963, 20000, 64, 256, 8),
        # the batched workload on the paper's 64-GPU Cascadia grid: 256 ruptures, uneven durations
        _case("bf16_b256_active", "active", "bf16", "bf16", 963, 37758, 64, 256, 256),
        # one sub-batch of the largest workload's kind: FP8 operators, the default precision of the benchmark
        _case("fp8_b256", "waveforms", "fp8", "bf16", 963, 50000, 64, 256, 256),
        # an ensemble at FP32-class accuracy on the tensor engine, ragged batch and grid
        _case("hilo_b100", "waveforms", "bf16_hilo", "fp32", 963, 10007, 64, 256, 100),
        # the gradient workload: 64 ruptures, misfit gradient on transposed operator copies
        _case("gradient_hilo_b64", "gradient", "bf16_hilo", "fp32", 963, 8000, 64, 256, 64, True),
        # inversion at the default precision through autograd, odd sizes
        _case("autograd_fp32_b6", "autograd", "fp32", "fp32", 501, 10007, 33, 128, 6),
        # seafloor fields of a few ruptures, long records, odd sizes
        _case("seafloor_fp32_b5", "seafloor", "fp32", "fp32", 333, 4999, 17, 512, 5),
        # the transforms alone: the slip rows of 256 ruptures
        _case("transforms", "transforms", "fp32", "fp32", 963, 64, 2, 256, 256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["waveforms", "waveforms", "waveforms", "active", "seafloor", "gradient", "autograd", "transforms"])
    if op == "transforms":
        return {k: v for k, v in _case("", op, "fp32", "fp32", _log(rng, 16, 1000), 64, 2,
                                       rng.choice([32, 64, 128, 256, 512]), _log(rng, 1, 128)).items() if k != "name"}
    prec = rng.choice(["fp32", "fp32", "bf16", "bf16_hilo", "fp8", "fp32_hilo"])
    adj = False
    if op in ("gradient", "autograd"):
        prec = rng.choice(["fp32", "fp32", "bf16", "bf16_hilo"])
        adj = prec != "fp32" and rng.random() < 0.5
    if op == "seafloor" and prec == "fp32_hilo":
        prec = "fp32"
    tensor = prec in ("bf16", "bf16_hilo", "fp8") and op != "seafloor" and (op not in ("gradient", "autograd") or adj)
    prec_p = {"fp32": "fp32", "fp32_hilo": "fp32_hilo", "bf16": "bf16", "fp8": "bf16",
              "bf16_hilo": "fp32"}[prec]
    Nt = rng.choice([64, 128, 256]) if tensor or prec == "fp32_hilo" else rng.choice([32, 64, 128, 256, 512])
    Ns, No = _log(rng, 8, 1024), _log(rng, 2, 120)
    B = _log(rng, 1, 256) if tensor else (_log(rng, 1, 3) if prec == "fp32_hilo" else _log(rng, 1, 12))
    # at most ~6 GB of FP32 spectra, less where the batch (and so the time) is large
    most = max(600, min(16000, int(6e9 / ((Nt + 1) * 8 * Ns) / (1 if B <= 12 else 2))))
    Ng = _log(rng, 400, most)
    return {k: v for k, v in _case("", op, prec, prec_p, Ns, Ng, No, Nt, B, adj).items() if k != "name"}


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
class _Scene:
    """Fault plane, grid and observations of one (case, seed)."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([int(seed), case["Ns"], case["Ng"], case["No"], case["Nt"]])
        Ns, Ng, No = case["Ns"], case["Ng"], case["No"]
        length = 1000.0 * case["Nt"] / 256.0  # the record covers the same share of the fault at every length
        dip = math.radians(12.0)
        u, w = rng.uniform(0, length, Ns), rng.uniform(0, 100.0, Ns)
        self.length, self.rng, self.case = length, rng, case

        def dev(a):
            return torch.tensor(a, dtype=torch.float32, device=DEV)

        def surface(n):
            return dev(np.stack([rng.uniform(-50, length + 50, n), rng.uniform(-50, 148, n), np.zeros(n)], 1))
        self.sub = dev(np.stack([u, w * math.cos(dip), 5.0 + w * math.sin(dip)], 1))
        self.grid, self.obs = surface(Ng), surface(No)
        self.u, self.w = dev(u), dev(w)

    def _response(self, a, b, kms):
        d = torch.sqrt(((a[:, None, :] - b[None, :, :]) ** 2).sum(-1))
        t = torch.arange(self.case["Nt"], dtype=torch.float32, device=DEV) - (d / kms)[..., None]
        t = t.mul_(math.pi * F0_HZ).square_()
        r = torch.exp(-t)
        r.mul_(t.mul_(-2.0).add_(1.0))
        return r.mul_(torch.exp(-d / DECAY_KM)[..., None])

    def chunks(self, columns, bytes_per_value, most=2 << 30):
        """Grid row ranges (multiples of 256 rows) of at most `most` bytes for rows of `columns` x Nt values."""
        step = max(256, most // (columns * self.case["Nt"] * bytes_per_value) // 256 * 256)
        return [(i, min(i + step, self.case["Ng"])) for i in range(0, self.case["Ng"], step)]

    def greens(self, i0, i1):
        return self._response(self.grid[i0:i1], self.sub, GREEN_KMS)

    def adjoint(self, i0, i1):
        return self._response(self.obs, self.grid[i0:i1], ADJ_KMS)

    def slip(self):
        """[B][Ns][Nt] slip rates (m/s): patches of log-normal slip, triangular source-time functions."""
        B, Ns, Nt = self.case["B"], self.case["Ns"], self.case["Nt"]
        rng = self.rng

        def dev(a):
            return torch.tensor(a, dtype=torch.float32, device=DEV)
        hu, hw = dev(rng.uniform(0, self.length, B)), dev(rng.uniform(0, 100.0, B))
        ext = dev(rng.uniform(0.15, 0.6, B) * self.length)
        du, dw = (self.u[None] - hu[:, None]), (self.w[None] - hw[:, None])
        amp = dev(rng.lognormal(0.5, 0.8, (B, Ns)))
        amp = amp * torch.clamp(1.0 - (du / ext[:, None]) ** 2 - (dw / 80.0) ** 2, min=0.0)
        t0 = torch.sqrt(du * du + dw * dw) / RUPTURE_KMS
        half = 0.5 * torch.clamp(4.0 * torch.sqrt(amp), 3.0, 40.0)
        s = torch.arange(Nt, dtype=torch.float32, device=DEV) - (t0 + half)[..., None]
        s = s.abs_().div_(-half[..., None]).add_(1.0).clamp_(min=0.0)
        return s.mul_((amp / half)[..., None])

    def lens(self):
        return self.rng.integers(min(32, self.case["Nt"]), self.case["Nt"] + 1, self.case["B"]).astype(np.int32)

    def targets(self):
        """[B][No][Nt] observed waveforms: a few pulses per record, as large as the operators' waveforms are."""
        B, No, Nt = self.case["B"], self.case["No"], self.case["Nt"]
        rng = self.rng
        t = torch.arange(Nt, dtype=torch.float32, device=DEV)
        d = torch.zeros(B, No, Nt, device=DEV)
        for _ in range(3):
            t0 = torch.tensor(rng.uniform(0, Nt, (B, No, 1)), dtype=torch.float32, device=DEV)
            a = torch.tensor(rng.standard_normal((B, No, 1)), dtype=torch.float32, device=DEV)
            x = (math.pi * 0.05 * (t - t0)) ** 2
            d += a * (1 - 2 * x) * torch.exp(-x)
        return d * (0.1 * self.case["Ng"])


def _context(case):
    c = case
    return s2w.Context(c["Ns"], c["Ng"], c["No"], c["Nt"], prec_g=c["prec_g"], prec_p=c["prec_p"], max_batch=c["B"],
                       tc_adjoint=c["tc_adjoint"])


def prepare(case, seed):
    if case["op"] == "transforms":
        rows = case["B"] * case["Ns"]
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        x = torch.randn(rows, case["Nt"], generator=gen, device=DEV)
        return {"op": "transforms", "ctx": s2w.Context(8, 64, 2, case["Nt"]), "x": x}
    sc = _Scene(case, seed)
    state = {"op": case["op"], "slip": sc.slip()}
    if case["op"] == "active":
        state["lens"] = sc.lens()
    if case["op"] in ("gradient", "autograd"):
        state["d"] = sc.targets()
    if case["op"] == "autograd":
        state["slip"].requires_grad_(True)
    if case["op"] == "seafloor":
        state["shape"] = (case["B"], case["Ng"], case["Nt"])
    ctx = state["ctx"] = _context(case)
    for i0, i1 in sc.chunks(case["Ns"], 4):
        ctx.load_greens(i0, sc.greens(i0, i1))
    for i0, i1 in sc.chunks(case["No"], 4):
        ctx.load_adjoint(i0, sc.adjoint(i0, i1))
    return state


def run(state):
    ctx, op = state["ctx"], state["op"]
    if op == "waveforms":
        return {"q": ctx.waveforms(state["slip"])}
    if op == "active":
        return {"q": ctx.waveforms_active(state["slip"], state["lens"])}
    if op == "seafloor":
        field = torch.empty(state["shape"], dtype=torch.float32, device=DEV)
        return {"q": ctx.waveforms(state["slip"], seafloor=field), "seafloor": field}
    if op == "gradient":
        grad, loss = ctx.misfit_gradient(state["slip"], state["d"])
        return {"grad": grad, "loss": loss}
    if op == "autograd":
        loss = autograd.misfit(ctx, state["slip"], state["d"])
        grad, = torch.autograd.grad(loss, state["slip"])
        return {"grad": grad, "loss": loss.detach()}
    X = ctx.rfft(state["x"])
    return {"X": X, "x": ctx.irfft(X)}


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
_COMPLEX = {"fp32": 8, "fp32_hilo": 16, "bf16": 4, "bf16_hilo": 8, "fp8": 2}


def work(case):
    Ns, Ng, No, Nt, B, Nb = case["Ns"], case["Ng"], case["No"], case["Nt"], case["B"], case["Nt"] + 1

    def fft(rows):  # a real FFT of length 2 Nt
        return rows * 2.5 * (2 * Nt) * math.log2(2 * Nt)
    if case["op"] == "transforms":
        rows = B * Ns
        return {"bytes": rows * (2 * 4 * Nt + 2 * 8 * Nb), "flops": 2 * fft(rows)}
    ops = Nb * Ng * (Ns * _COMPLEX[case["prec_g"]] + No * _COMPLEX[case["prec_p"]])
    rows = Ns + 2 * Ng + No
    n_bytes = ops + 4 * B * Nt * (Ns + No)
    flops = 8.0 * Nb * Ng * (Ns + No) * B + fft(B * rows)
    if case["op"] == "seafloor":
        n_bytes += 4 * B * Nt * Ng
    if case["op"] in ("gradient", "autograd"):
        # the adjoint needs the whole misfit, so the operators are read again
        n_bytes += ops + 4 * B * Nt * (No + Ns)
        flops *= 2
    return {"bytes": n_bytes, "flops": flops}


# --------------------------------------------------------------------------
# The same in 64 bits
# --------------------------------------------------------------------------
def _rfft(x, Nt):
    return torch.fft.rfft(x.double(), n=2 * Nt)


def _head(X, Nt):
    return torch.fft.irfft(X, n=2 * Nt)[..., :Nt]


def exact(case, seed):
    Nt, B = case["Nt"], case["B"]
    if case["op"] == "transforms":
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        x = torch.randn(B * case["Ns"], Nt, generator=gen, device=DEV)
        return {"X": _rfft(x, Nt), "x": x.double()}
    if 8.0 * (Nt + 1) * case["Ng"] * (case["Ns"] + case["No"]) * B > 8e12:
        return None  # over about 20 s of 64-bit arithmetic
    sc = _Scene(case, seed)
    slip = sc.slip()
    if case["op"] == "active":
        n = torch.arange(Nt, device=DEV)
        slip = slip * (n[None, None] < torch.tensor(sc.lens(), device=DEV)[:, None, None])
    d = sc.targets().double() if case["op"] in ("gradient", "autograd") else None
    shat = _rfft(slip, Nt).permute(2, 1, 0).contiguous()  # [Nb][Ns][B]
    qhat = torch.zeros(Nt + 1, case["No"], B, dtype=torch.complex128, device=DEV)
    field = torch.empty(B, case["Ng"], Nt, dtype=torch.float64, device=DEV) if case["op"] == "seafloor" else None
    parts = sc.chunks(max(case["Ns"], case["No"], B), 8, 1 << 30)
    for i0, i1 in parts:
        Gh = _rfft(sc.greens(i0, i1), Nt).permute(2, 0, 1).contiguous()  # [Nb][rows][Ns]
        m = _head(torch.bmm(Gh, shat).permute(2, 1, 0).contiguous(), Nt)  # [B][rows][Nt]
        del Gh
        if field is not None:
            field[:, i0:i1] = m
        v = torch.diff(m, dim=-1, prepend=torch.zeros_like(m[..., :1]))
        vhat = _rfft(v, Nt).permute(2, 1, 0).contiguous()
        Ph = _rfft(sc.adjoint(i0, i1), Nt).permute(2, 0, 1).contiguous()  # [Nb][No][rows]
        qhat += torch.bmm(Ph, vhat)
    q = _head(qhat.permute(2, 1, 0).contiguous(), Nt)
    if d is None:
        return {"q": q} if field is None else {"q": q, "seafloor": field}
    r = q - d
    rhat = _rfft(r, Nt).permute(2, 1, 0).contiguous()  # [Nb][No][B]
    ghat = torch.zeros(Nt + 1, case["Ns"], B, dtype=torch.complex128, device=DEV)
    for i0, i1 in parts:
        Ph = _rfft(sc.adjoint(i0, i1), Nt).permute(2, 1, 0).conj().resolve_conj().contiguous()  # [Nb][rows][No]
        w = _head(torch.bmm(Ph, rhat).permute(2, 1, 0).contiguous(), Nt)
        u = w - torch.cat([w[..., 1:], torch.zeros_like(w[..., :1])], -1)
        uhat = _rfft(u, Nt).permute(2, 1, 0).contiguous()
        Gh = _rfft(sc.greens(i0, i1), Nt).permute(2, 1, 0).conj().resolve_conj().contiguous()  # [Nb][Ns][rows]
        ghat += torch.bmm(Gh, uhat)
    grad = _head(ghat.permute(2, 1, 0).contiguous(), Nt)
    loss = 0.5 * (r * r).sum((1, 2))
    return {"grad": grad, "loss": loss.sum() if case["op"] == "autograd" else loss}
