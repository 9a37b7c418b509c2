"""Set-up calls have finished on the device when they return: the tables they
build are read by steps on whatever stream the context is given next, by the
first kernel of a step before its dependency wait, and by sadi_step_noalloc,
which needs no sadi_set_initial."""
import numpy as np
import pytest

from paper_2312_06206_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_06206_gb300 import build
    build.build()
    from paper_2312_06206_gb300 import sadi
    return sadi, torch


@pytest.mark.parametrize("N", [1, 63, 128])
def test_precision_switched_back_to_fp64_leaves_no_pending_work(env, N):
    # FP64 -> FP32 -> FP64 rebuilds the dense tables of the small FP64 step
    S, torch = env
    setup, other = torch.cuda.Stream(), torch.cuda.Stream()
    phi = WL.gaussian_bumps(N, 4, 4000 + N)
    out = []
    for switch in (False, True):
        with S.Sadi(N, 1.6, 1.0, 0.2 / (N + 1)) as s:
            s.set_stream(setup.cuda_stream)
            s.set_options(1, S.SADI_PREC_FP64)
            if switch:
                s.set_options(1, S.SADI_PREC_FP32)
                s.set_options(1, S.SADI_PREC_FP64)
                assert setup.query()
            s.set_stream(other.cuda_stream)
            u = [torch.from_numpy(a).cuda() for a in (phi, phi, np.zeros_like(phi))]
            torch.cuda.synchronize()
            s.sadi_step_noalloc(u[0].data_ptr(), u[1].data_ptr(), u[2].data_ptr(), 1)
            s.set_initial(phi)
            s.step(3)
            out.append((s.get()[0], u[2].cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_three_pass_convolution_set_up_leaves_no_pending_work(env):
    # explicit tiles with conv_cols = -1 build the symbol table of the three
    # passes (134 MB at N' = 4096)
    S, torch = env
    setup = torch.cuda.Stream()
    with S.Sadi(4090, 1.6, 1.0, 1e-4) as s:
        s.set_stream(setup.cuda_stream)
        s.set_options(1, S.SADI_PREC_FP32)
        s.sadi_set_tiles(1, -1, 1)
        assert setup.query()
