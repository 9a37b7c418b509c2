"""sadi_step_source reads a float field of the step's precision in place on
every engine of the FP32 forms: no copy into a buffer of the context (which the
first such call would allocate), and the bits of the same field converted from
double (which does go through that buffer, at the padded row pitch)."""
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
    yield sadi, torch
    torch.cuda.empty_cache()      # later tests measure and bound allocations


@pytest.mark.parametrize("equation", ["wave", "diffusion"])
@pytest.mark.parametrize("N,prec_name,tiles", [(255, "SADI_PREC_FP32", False), (2047, "SADI_PREC_FP32", False),
                                               (2047, "SADI_PREC_FP32_DENSE", True),
                                               (4090, "SADI_PREC_FP32_DENSE", False)])
def test_float_source_is_read_in_place(env, N, prec_name, tiles, equation):
    S, torch = env
    f = torch.from_numpy(0.3 * WL.gaussian_bumps(N, 2, 4700 + N)).to("cuda").float()
    g = f.double()
    torch.cuda.synchronize()
    tau = 0.2 / (N + 1) if equation == "wave" else 0.02 / (N + 1) ** 1.4
    out = []
    for field, dtype in ((f, 1), (g, 0)):
        with S.Sadi(N, 1.4, 0.9, tau, equation=equation) as s:
            s.set_options(1, getattr(S, prec_name))
            if tiles:
                s.sadi_set_tiles(*s.sadi_get_tiles())
            s.set_initial(WL.gaussian_bumps(N, 4, 4800 + N))
            s.step(1)                       # everything a step itself loads or allocates
            s.sadi_wait()
            before = torch.cuda.mem_get_info()[0]
            for _ in range(2):
                s.sadi_step_source(field.data_ptr(), dtype)
            s.sadi_wait()
            grown = before - torch.cuda.mem_get_info()[0]
            assert dtype == 0 or grown < 4 * N * N, grown
            out.append(s.get()[0])
    assert np.array_equal(out[0], out[1])
