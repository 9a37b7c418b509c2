"""FP64 at N <= 128 over many steps.  The dense products of the small FP64 step
took the place of transforms for their speed alone, so they may be no further
from the scheme than the transforms are (tiles other than the defaults).

A table that is a unit in the last place off is the same error in every step,
and the leapfrog adds it up twice: three steps cannot show it, 200 do.  The
reference is the scheme in extended precision (np.longdouble) on the library's
own weights a_i and a_ij: symbol and FFTs, state, remainder and the inverse of
I + s T all carry 2^-63 or less, which keeps it within 1e-16 of the field.

Tolerance: both step forms round the same state in the same places, which sets
the error they cannot go below, and their maxima over 4000 to 16000 values of
independent rounding errors differ by less than a factor of two."""
import math

import numpy as np
import pytest

from paper_2312_06206_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_06206_gb300 import build
    build.build()
    from paper_2312_06206_gb300 import sadi
    return sadi


def _cos_table(M, n, rows):
    """cos(2 pi i k / M), i < rows, k < n, from angles in [0, pi / 4]"""
    pi = 4 * np.arctan(L(1))
    m = np.arange(M // 2 + 1)
    q = np.minimum(m, M // 2 - m)
    c = np.where(8 * q <= M, np.cos(2 * pi * q / M), np.sin(2 * pi * (M // 4 - q) / M))
    c = np.where(4 * m <= M, c, -c)
    return np.concatenate([c, c[-2:0:-1]])[np.outer(np.arange(rows), np.arange(n)) % M]


def _reference(a1, a2, s, tau, phi, steps):
    """u^steps of the wave scheme with g = -u^3, phi2 = 0; a2[dx, dy]"""
    import scipy.fft as sf
    N = len(a1)
    P = 4
    while P < 2 * N:
        P *= 2
    C = _cos_table(P, N, P // 2 + 1)
    C[:, 1:] *= 2
    lam = -2 * L(s) * (C @ a2.T.astype(L) @ C.T)
    lam = np.concatenate([lam, lam[-2:0:-1]], 0)
    i = np.arange(N)
    T = L(s) * a1.astype(L)[np.abs(i[:, None] - i[None, :])]
    X = np.linalg.inv((T + np.eye(N)).astype(np.float64)).astype(L) - np.eye(N)
    R = -(X + T + T @ X)
    E = X + R + X @ R
    E0 = E.astype(np.float64)
    E1 = (E - E0).astype(np.float64)

    def conv(d):
        return sf.irfft2(sf.rfft2(d, s=(P, P)) * lam, s=(P, P))[:N, :N]

    def sweep(b):
        b64 = b.astype(np.float64)
        return b + (b64 @ E0) + (b64 @ E1)

    t2 = L(tau) * L(tau)
    u = phi.astype(L)
    d = np.zeros_like(u)
    c = conv(u)
    for n in range(steps):
        b = c - t2 * u * u * u
        d = d + sweep(sweep(b / 2 if n == 0 else b).T).T
        u = u + d
        c = c + conv(d)
    return u


@pytest.mark.parametrize("N,alpha,steps", [(63, 1.5, 200), (63, 1.9, 200), (127, 1.5, 60), (128, 1.9, 60)])
def test_small_fp64_step_stays_as_exact_as_the_transforms(S, N, alpha, steps):
    h = 2.0 / (N + 1)
    tau = 0.35 * h
    s_adi = tau * tau / (2.0 * math.pow(h, alpha))
    phi = WL.gaussian_bumps(N, 8, 4600 + N)
    u = []
    for tiles in (False, True):
        with S.Sadi(N, alpha, 1.0, tau) as s:
            s.set_options(S.SADI_G_NEG_CUBE, S.SADI_PREC_FP64)
            if tiles:
                t = s.sadi_get_tiles()
                s.sadi_set_tiles(t[0] + 1, t[1], t[2])
            a1, a2 = s.sadi_get_setup(0).reshape(-1), s.sadi_get_setup(1).reshape(N, N)
            s.set_initial(phi)
            s.step(steps)
            u.append(s.get()[0])
    ref = _reference(a1, a2, s_adi, tau, phi, steps)
    dense, transforms = (float(np.abs(v - ref).max() / np.abs(ref).max()) for v in u)
    assert dense <= 2.0 * transforms, (dense, transforms)
