"""The work whose speed matters to users of this library, as cases that can be timed.

A case is one stretch of time steps of one problem, or of many independent
problems together, from the state that a program holds to the field that it
reads back: `prepare` creates the contexts, sets the initial data and takes the
first step; `run` advances them and copies the new fields into device tensors
of the caller's.  Everything runs on one stream, as in a program that drives
one simulation.

Families (the "kind" of a case):
  single     one wave-equation context, Sadi.step
  replay     several contexts of one size, their batched step replayed as a
             captured graph (SadiGraph), as the throughput runs do
  mixed      contexts of uneven N, alpha and kappa in one replayed batch
  diffusion  one diffusion context driven by a source field, a step at a time

`exact` is the same scheme in 64-bit torch: trapezoid-rule weights with one
Richardson step, the L_h product by zero-padded 2D FFTs, and the Toeplitz
solves by a converged fixed-point iteration or a dense inverse.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2312_06206_gb300 import sadi as S

PREC = {"fp64": S.SADI_PREC_FP64, "fp32": S.SADI_PREC_FP32, "dense": S.SADI_PREC_FP32_DENSE}
G_KINDS = {"zero": S.SADI_G_ZERO, "cube": S.SADI_G_NEG_CUBE, "sin": S.SADI_G_NEG_SIN, "general": S.SADI_G_GENERAL}
GENERAL = (-1.0, -0.5, 0.25)        # c1, c3, cs of the "general" nonlinearity

_stream = None


def stream():
    """The program's stream: every context issues its work here."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def case(name, kind, prec, N, steps, alpha=1.5, kappa=1.0, tau=1e-3, half=1.0, g="sin", bumps=8, phi2=0.0, count=1,
         mix=0):
    """half: the domain is (-half, half)^2; phi2: initial velocity phi2 * phi1;
    count: contexts; mix: seed of the members' sizes and parameters."""
    d = dict(kind=kind, prec=prec, N=N, steps=steps, alpha=alpha, kappa=kappa, tau=tau, half=half, g=g, bumps=bumps,
             phi2=phi2, count=count, mix=mix)
    return dict(d, name=name) if name else d


def listed():
    return [
        # a small problem in the default precision: 63 points per direction,
        # tau = 1/64, -u^3; every kernel is short, so launches and latency count
        case("fp64-n63", "single", "fp64", 63, 16, 1.5, 1.0, 1 / 64, g="cube", bumps=1),
        # the grids of the published tables on (-10, 10)^2, which are not one
        # below a power of two: h = 1/40 (N = 799) in FP64 and h = 1/20
        # (N = 399) in FP32
        case("fp64-n799", "single", "fp64", 799, 2, 1.5, 1.0, 1 / 80, half=10.0, g="sin", phi2=1.0),
        case("fp32-n399", "single", "fp32", 399, 8, 1.5, 1.0, 1 / 125, half=10.0, g="cube"),
        # plain FP64 at the benchmark size: the accuracy reference that the
        # FP32 forms are compared with
        case("fp64-n1023", "single", "fp64", 1023, 2, 1.5, 1.0, 1e-3, g="sin"),
        # one FP32 problem of the benchmark size, stepped directly
        case("fp32-n1023", "single", "fp32", 1023, 8, 1.8, 1.0, 1e-3, g="sin"),
        # the benchmark workload: three instances of N = 1023 in the dense-inverse
        # form, their batched step replayed from a graph
        case("dense-n1023x3", "replay", "dense", 1023, 8, 1.5, 1.0, 1e-3, g="sin", count=3),
        # the large precision workload, N = 4095, in both FP32 forms
        case("dense-n4095", "single", "dense", 4095, 2, 1.7, 0.5, 5e-4, g="cube"),
        case("fp32-n4095", "single", "fp32", 4095, 2, 1.7, 0.5, 5e-4, g="cube"),
        # the largest single instance, 67 M unknowns
        case("fp32-n8191", "single", "fp32", 8191, 1, 1.6, 1.0, 2.5e-4, g="sin", bumps=32, phi2=0.1),
        # many independent instances of N in {127 .. 2047}, each size in the
        # form that the autotuner picks for it
        case("mixed-x24", "mixed", "auto", 2047, 2, g="cube", count=24, mix=20231210),
        # a driven diffusion problem, a new source every step
        case("diffusion-n255", "diffusion", "fp32", 255, 8, 1.5, 1.0, 1e-2, g="general"),
    ]


def draw(rng):
    kind = rng.choice(["single", "single", "single", "replay", "mixed", "diffusion"])
    alpha, kappa = round(rng.uniform(1.1, 1.9), 3), round(rng.uniform(0.5, 2.0), 3)
    g = rng.choice(["zero", "cube", "sin", "general"])
    bumps = rng.randint(1, 16)
    if kind == "mixed":
        return case(None, kind, "auto", 2047, rng.randint(1, 3), g=g, bumps=bumps, count=rng.randint(4, 24),
                    mix=rng.randrange(1 << 30))
    prec = rng.choice(["fp32", "dense"]) if kind == "replay" else rng.choice(["fp64", "fp32", "dense"])
    if kind == "diffusion":
        prec = rng.choice(["fp64", "fp32"])
    top = {"single": {"fp64": 2048, "fp32": 8192, "dense": 4096}[prec], "replay": 1024, "diffusion": 1024}[kind]
    N = int(round(math.exp(rng.uniform(math.log(24), math.log(top)))))
    if rng.random() < 0.4:
        N = (1 << max(5, N.bit_length() - 1)) - 1         # one below a power of two
    elif N > 4096:
        N = 8191
    elif N > 1024:
        # the set-up's border solve grows with the cube of the distance to the
        # next power of two, so large grids in use lie close below one
        N = min(1 << N.bit_length(), top) - rng.randint(0, 64)
    h = 2.0 / (N + 1)
    tau = h * rng.uniform(0.1, 0.25) if prec == "dense" else h * rng.uniform(0.2, 0.5)
    count = rng.randint(2, 8) if kind == "replay" else 1
    steps = 1 if N > 2100 else rng.randint(1, 4) if N > 700 else rng.randint(4, 12)
    return case(None, kind, prec, N, steps, alpha, kappa, tau, g=g, bumps=bumps,
                phi2=0.0 if kind == "diffusion" else rng.choice([0.0, 0.1]), count=count)


def members(c):
    """The problems of a case: dicts of N, alpha, kappa, tau, prec."""
    if c["kind"] == "mixed":
        r = random.Random(c["mix"])
        out = []
        for _ in range(c["count"]):
            N = r.choice([127, 255, 511, 1023, 2047])
            # tau = h/4 keeps every member inside the dense form's accuracy range
            out.append(dict(N=N, alpha=r.uniform(1.1, 1.9), kappa=r.uniform(0.5, 2.0), tau=0.5 / (N + 1),
                            prec="fp32" if N <= 255 else "dense"))
        return out
    one = {k: c[k] for k in ("N", "alpha", "kappa", "tau", "prec")}
    if c["kind"] == "replay":
        # the instances differ in alpha
        return [dict(one, alpha=min(1.9, max(1.1, c["alpha"] + 0.3 * (k - 1)))) for k in range(c["count"])]
    return [one]


def initial(N, half, bumps, seed):
    """A sum of Gaussian bumps: centres U(-0.6, 0.6), widths U(0.05, 0.2) (of
    the half width), amplitudes U(-1, 1)."""
    r = np.random.default_rng(seed)
    x = (-1.0 + 2.0 / (N + 1) * np.arange(1, N + 1))[None, :]
    cx, cy = r.uniform(-0.6, 0.6, (bumps, 1)), r.uniform(-0.6, 0.6, (bumps, 1))
    w, a = r.uniform(0.05, 0.2, (bumps, 1)), r.uniform(-1.0, 1.0, (bumps, 1))
    ex, ey = np.exp(-((x - cx) ** 2) / (2 * w * w)), np.exp(-((x - cy) ** 2) / (2 * w * w))
    return np.ascontiguousarray((a * ey).T @ ex)


def source(c, seed):
    """The diffusion case's source field, in the type of the context's step."""
    return initial(c["N"], 1.0, 4, seed + 7919).astype(np.float64 if c["prec"] == "fp64" else np.float32)


def fields(c, m, k, seed):
    phi1 = initial(m["N"], c["half"], c["bumps"], seed * 131 + k)
    return phi1, (c["phi2"] * phi1 if c["phi2"] else None)


def prepare(c, seed):
    st, ctxs, outs = stream(), [], []
    eq = "diffusion" if c["kind"] == "diffusion" else "wave"
    f = None
    if eq == "diffusion":
        f = torch.from_numpy(source(c, seed)).cuda()
    torch.cuda.synchronize()
    for k, m in enumerate(members(c)):
        s = S.Sadi(m["N"], m["alpha"], m["kappa"], m["tau"], (-c["half"], c["half"]), equation=eq)
        s.set_stream(st.cuda_stream)
        s.set_options(G_KINDS[c["g"]], PREC[m["prec"]])
        if c["g"] == "general":
            s.sadi_set_nonlinearity(*GENERAL)
        phi1, phi2 = fields(c, m, k, seed)
        s.set_initial(phi1, phi2)
        ctxs.append(s)
        outs.append(torch.zeros((m["N"], m["N"]), dtype=torch.float64 if m["prec"] == "fp64" else torch.float32,
                                device="cuda"))
    graph = None
    if f is not None:
        ctxs[0].sadi_step_source(f.data_ptr(), int(f.dtype == torch.float32))
    else:
        S.sadi_batch_step(ctxs, 1)
    if c["kind"] in ("replay", "mixed"):
        graph = S.SadiGraph(ctxs)
    torch.cuda.synchronize()
    return dict(kind=c["kind"], steps=c["steps"], graph=graph, ctxs=ctxs, outs=outs, f=f)


def run(state):
    ctxs = state["ctxs"]
    if state["graph"] is not None:
        state["graph"].launch(state["steps"])
    elif state["f"] is not None:
        f = state["f"]
        for _ in range(state["steps"]):
            ctxs[0].sadi_step_source(f.data_ptr(), int(f.dtype == torch.float32))
    else:
        ctxs[0].step(state["steps"])
    for s, o in zip(ctxs, state["outs"]):
        s.sadi_get_device(o.data_ptr(), 0 if o.dtype == torch.float64 else 1)
    return state["outs"]


def work(c):
    b = f = 0.0
    for m in members(c):
        n2, es = float(m["N"]) ** 2, 8 if m["prec"] == "fp64" else 4
        # a step reads u^n and u^{n-1} and writes u^{n+1}; the field is read
        # and written once more for the caller.  The transforms of a step: 1 of
        # length N' per row, 4 per column, 1 + 4 per row and 4 per column
        # (5 L log2 L operations each)
        b += n2 * es * (3 * c["steps"] + 2)
        f += n2 * c["steps"] * 70.0 * math.log2(max(8, m["N"]))
    return {"bytes": b, "flops": f}


# ---- the scheme in 64 bits ------------------------------------------------------


def weights_1d(alpha, n):
    a = [math.gamma(alpha + 1.0) / math.gamma(alpha / 2.0 + 1.0) ** 2]
    for i in range(n - 1):
        a.append(a[-1] * (i - alpha / 2.0) / (i + 1.0 + alpha / 2.0))
    return torch.tensor(a, dtype=torch.float64, device="cuda")


def even_dft(x, n):
    """sum_k f_k cos(2 pi i k / M), i < n, of the even sequence whose half
    f_0 .. f_{M/2} is x, along the last dimension."""
    M = 2 * (x.shape[-1] - 1)
    return torch.fft.irfft(x.to(torch.complex128), n=M, dim=-1)[..., :n] * M


def weights_2d(alpha, N, Np):
    def trap(M):
        half = M // 2 + 1
        s = 4.0 * torch.sin(math.pi * torch.arange(half, dtype=torch.float64, device="cuda") / M) ** 2
        rows = max(1, (1 << 28) // (2 * M))
        T = torch.empty((half, N), dtype=torch.float64, device="cuda")
        for r in range(0, half, rows):
            T[r:r + rows] = even_dft((s[r:r + rows, None] + s[None, :]) ** (alpha / 2.0), N)
        T = T.t().contiguous()
        A = torch.empty((N, N), dtype=torch.float64, device="cuda")
        for r in range(0, N, rows):
            A[r:r + rows] = even_dft(T[r:r + rows], N)
        return A / float(M) ** 2
    M = max(1024, 8 * Np)
    q = 2.0 ** (2.0 + alpha)
    return (q * trap(2 * M) - trap(M)) / (q - 1.0)


def wrapped(a, P, dims):
    """a_|i| at i mod P (zero beyond), along each of the dims."""
    for d in dims:
        n = a.shape[d]
        pad = list(a.shape)
        pad[d] = P - 2 * n + 1
        tail = a.narrow(d, 1, n - 1).flip(d)
        a = torch.cat([a, a.new_zeros(pad), tail], dim=d)
    return a


class Exact:
    def __init__(self, m, half, eq):
        N = self.N = m["N"]
        Np = 8
        while Np < N:
            Np *= 2
        self.P, h, al = 2 * Np, 2.0 * half / (N + 1), m["alpha"]
        self.tau, self.tp = m["tau"], m["tau"] ** 2 if eq == "wave" else m["tau"]
        self.s = m["kappa"] * self.tp / (2.0 * h ** al)
        a1 = weights_1d(al, N)
        self.k1 = torch.fft.rfft(wrapped(a1, self.P, [0])).real
        # the factor kappa tp h^-alpha of L_h is 2 s
        self.k2 = torch.fft.rfft2(wrapped(weights_2d(al, N, Np), self.P, [0, 1])).real
        self.top = self.s * 2.0 ** al                     # the eigenvalues of sT lie in (0, top]
        self.inv = None
        if self.top > 1.5:
            idx = torch.arange(N, device="cuda")
            self.inv = torch.linalg.inv(torch.eye(N, dtype=torch.float64, device="cuda")
                                        + self.s * a1[(idx[:, None] - idx[None, :]).abs()])

    def lap(self, u):
        """kappa tp L_h u"""
        N, P = self.N, self.P
        return 2.0 * self.s * torch.fft.irfft2(torch.fft.rfft2(u, s=(P, P)) * self.k2, s=(P, P))[:N, :N]

    def solve_rows(self, b):
        if self.inv is not None:
            return b @ self.inv
        w, x = 2.0 / (2.0 + self.top), torch.zeros_like(b)
        rate = self.top / (2.0 + self.top)
        for _ in range(max(2, int(math.ceil(-39.0 / math.log(rate))))):
            t = torch.fft.irfft(torch.fft.rfft(x, n=self.P) * self.k1, n=self.P)[:, :self.N]
            x = x + w * (b - x - self.s * t)
        return x

    def sweeps(self, b):
        w = self.solve_rows(b)
        return self.solve_rows(w.t().contiguous()).t()


def g_exact(kind, u):
    c1, c3, cs = {"zero": (0, 0, 0), "cube": (0, -1, 0), "sin": (0, 0, -1), "general": GENERAL}[kind]
    return c1 * u + c3 * u ** 3 + cs * torch.sin(u)


def exact(c, seed):
    eq = "diffusion" if c["kind"] == "diffusion" else "wave"
    outs = []
    for k, m in enumerate(members(c)):
        E = Exact(m, c["half"], eq)
        phi1, phi2 = fields(c, m, k, seed)
        u = torch.from_numpy(phi1).cuda()
        v = torch.from_numpy(phi2).cuda() if phi2 is not None else torch.zeros_like(u)
        f = torch.from_numpy(source(c, seed)).cuda().double() if eq == "diffusion" else None
        d = torch.zeros_like(u)
        for n in range(c["steps"] + 1):
            if eq == "wave":
                b = -E.lap(u) + E.tp * g_exact(c["g"], u)
                if n == 0:
                    b = E.tau * v + 0.5 * b
                d = d + E.sweeps(b)
            else:
                w = u + 0.5 * d
                d = d + E.sweeps(-E.lap(w) + E.tp * (g_exact(c["g"], w) + f) - d)
            u = u + d
        outs.append(u)
        del E
    return outs
