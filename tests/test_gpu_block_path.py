"""The FP32 forms on the engines and lengths around the block-FFT path, which
serves FFT lengths 256 .. 1024 (GS form) and 256 .. 2048 (dense form), against
the shared-memory engine (explicit tiles), which runs the longer ones, and
against the FP64 path: at the smallest N of a length, N one above and below a
multiple of eight, border ranks around 32, and N = N' (no border).  Where a form
has one engine (GS from N' = 2048, dense from 4096 on) the two runs of the engine
comparisons are the same engine; batches of uneven border ranks at the lengths
that batch them are in test_gpu_batch_uneven.py.

Tolerances: both engines compute the same FP32 transforms in different orders.
One transform of length L carries a relative error of about eps log2 L
(6e-8 x 13 < 1e-6) and the increment it yields is at most tau ||u_t|| / ||u|| <
1e-1 of the field per step here, so three steps agree to 1e-6 of the largest
value; the FP32 forms' bound against FP64 is 1e-5."""
import numpy as np
import pytest

from paper_2312_06206_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_06206_gb300 import build
    build.build()
    from paper_2312_06206_gb300 import sadi
    return sadi


def _run(S, N, prec, equation, tiles=False, g=3):
    tau = 1e-3 if equation == "wave" else 3e-6
    phi1 = WL.gaussian_bumps(N, 6, 3000 + N)
    phi2 = 0.1 * WL.gaussian_bumps(N, 3, 3100 + N) if equation == "wave" else None
    with S.Sadi(N, 1.4, 0.9, tau, equation=equation) as s:
        s.sadi_set_nonlinearity(-1.0, -0.5, 0.25)
        s.set_options(g, prec)
        if tiles:
            s.sadi_set_tiles(*s.sadi_get_tiles())
        s.set_initial(phi1, phi2)
        s.step(3)
        return s.get()[0]


@pytest.mark.parametrize("N", [1025, 2015, 2016, 2041, 2048, 4089, 4095, 4096])
@pytest.mark.parametrize("equation", ["wave", "diffusion"])
@pytest.mark.parametrize("prec_name", ["SADI_PREC_FP32", "SADI_PREC_FP32_DENSE"])
def test_block_path_against_shared_memory_engine(S, N, equation, prec_name):
    prec = getattr(S, prec_name)
    u = _run(S, N, prec, equation)
    v = _run(S, N, prec, equation, tiles=True)
    # the block path is the default for the dense form at N' = 2048 only; else
    # explicit tiles equal to the defaults are the same engine
    two = prec == S.SADI_PREC_FP32_DENSE and N <= 2048
    assert np.array_equal(u, v) != two
    assert np.abs(u - v).max() <= 1e-6 * np.abs(v).max()
    if N in (1025, 2015, 2048):
        w = _run(S, N, S.SADI_PREC_FP64, equation)
        assert np.abs(u - w).max() <= 1e-5 * np.abs(w).max()


def test_block_path_batch_of_uneven_border_ranks(S):
    # one launch per kernel for members of N' = 2048 with r = 1, 33 and 0;
    # bitwise what each gives alone
    Ns = [2047, 2015, 2048]
    phis = [WL.gaussian_bumps(N, 4, 3200 + N) for N in Ns]

    def make():
        out = []
        for N, p in zip(Ns, phis):
            s = S.Sadi(N, 1.5, 1.0, 1e-3)
            s.set_options(1, S.SADI_PREC_FP32)
            s.set_initial(p)
            out.append(s)
        return out
    alone, batch = make(), make()
    for s in alone:
        s.step(3)
    S.sadi_batch_step(batch, 3)
    for a, b in zip(alone, batch):
        assert np.array_equal(a.get()[0], b.get()[0])
        a.close()
        b.close()


def test_tiles_move_a_running_context_between_the_engines(S):
    # tiles set and cleared between steps: the GS form at N' = 2048 has one
    # engine, so nothing changes
    N = 1100
    phi1 = WL.gaussian_bumps(N, 4, 3300)
    us = []
    for switch in (False, True):
        with S.Sadi(N, 1.5, 1.0, 1e-3) as s:
            s.set_options(1, S.SADI_PREC_FP32)
            s.set_initial(phi1)
            s.step(2)
            if switch:
                s.sadi_set_tiles(*s.sadi_get_tiles())
            s.step(2)
            if switch:
                s.sadi_set_tiles(0, 0, 0)
            s.step(1)
            us.append(s.get()[0])
    assert np.array_equal(us[0], us[1])


def _small(S, N, prec, equation, tiles=False, source=False):
    tau = 0.2 / (N + 1) if equation == "wave" else 0.02 / (N + 1) ** 1.4
    phi1 = WL.gaussian_bumps(N, 5, 3400 + N)
    phi2 = 0.1 * WL.gaussian_bumps(N, 3, 3500 + N) if equation == "wave" else None
    with S.Sadi(N, 1.4, 0.9, tau, equation=equation) as s:
        s.set_options(2, prec)
        if tiles:
            t = s.sadi_get_tiles()
            s.sadi_set_tiles(t[0] + 1, t[1], t[2])
        s.set_initial(phi1, phi2)
        if source:
            import torch
            f = torch.from_numpy(0.3 * WL.gaussian_bumps(N, 2, 3600 + N)).to("cuda").float()
            for _ in range(3):
                s.sadi_step_source(f.data_ptr(), 1)
        else:
            s.step(3)
        return s.get()[0]


@pytest.mark.parametrize("N", [65, 95, 96, 128, 129, 223, 224, 255, 256, 257, 479, 480, 511, 512, 513, 991, 992, 1023])
@pytest.mark.parametrize("equation", ["wave", "diffusion"])
def test_small_fp32_paths_against_fp64(S, N, equation):
    # N' = 128 .. 1024: eight or four rows a block, the border correction added
    # in the sweeps (r <= 32), by dense sweeps (N' <= 512) or by the separate
    # product (N' = 1024); with and without a caller's source field (rows of N)
    for source in (False, True):
        w = _small(S, N, S.SADI_PREC_FP64, equation, source=source)
        for prec in (S.SADI_PREC_FP32, S.SADI_PREC_FP32_DENSE):
            u = _small(S, N, prec, equation, source=source)
            assert np.abs(u - w).max() <= 1e-6 * np.abs(w).max(), (prec, source)


@pytest.mark.parametrize("N", [1, 2, 5, 31, 63, 64, 65, 100, 127, 128])
@pytest.mark.parametrize("equation", ["wave", "diffusion"])
def test_small_fp64_step_against_the_transforms(S, N, equation):
    # the direct path (dense products, the default up to N' = 128) against the
    # shared-memory engine (tiles other than the defaults): at most 8 N' + 2 products are
    # summed per value, 1e-16 x sqrt(1000) x 3 steps < 1e-13 of the largest
    u = _small(S, N, S.SADI_PREC_FP64, equation)
    v = _small(S, N, S.SADI_PREC_FP64, equation, tiles=True)
    assert np.abs(u - v).max() <= 1e-13 * np.abs(v).max()


@pytest.mark.parametrize("N", [100, 300, 1023])
def test_source_field_off_its_alignment_is_copied(S, N):
    # a float field at an odd address is copied before the step reads it; the
    # same field on its alignment is read in place: the same bits
    import torch
    f = torch.from_numpy(0.3 * WL.gaussian_bumps(N, 2, 3700 + N)).to("cuda").float()
    buf = torch.zeros(4 * N * N + 16, dtype=torch.uint8, device="cuda")
    buf[2:2 + 4 * N * N] = f.reshape(-1).view(torch.uint8)
    torch.cuda.synchronize()
    out = []
    for p in (f.data_ptr(), buf.data_ptr() + 2):
        with S.Sadi(N, 1.4, 0.9, 0.2 / (N + 1)) as s:
            s.set_options(1, S.SADI_PREC_FP32)
            s.set_initial(WL.gaussian_bumps(N, 4, 3800 + N))
            for _ in range(2):
                s.sadi_step_source(p, 1)
            out.append(s.get()[0])
    assert np.array_equal(out[0], out[1])
