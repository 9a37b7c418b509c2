"""sadi_step_source with fields off the alignment of their elements: rows of N
elements that are also the context's pitch (N a multiple of 32, and FP64), and
fields of the other type.  The field is copied before a kernel reads it, so the
step gives the bits of the same field on its alignment."""
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


@pytest.mark.parametrize("N", [63, 64, 96, 1024, 1100])
@pytest.mark.parametrize("prec_name", ["SADI_PREC_FP64", "SADI_PREC_FP32"])
@pytest.mark.parametrize("dtype", [0, 1])
def test_misaligned_source_equals_aligned(env, N, prec_name, dtype):
    S, torch = env
    es = 8 if dtype == 0 else 4
    f = torch.from_numpy(0.3 * WL.gaussian_bumps(N, 2, 4400 + N)).to("cuda")
    f = f if dtype == 0 else f.float()
    buf = torch.zeros(es * N * N + 16, dtype=torch.uint8, device="cuda")
    off = es // 2 + 1
    buf[off:off + es * N * N] = f.reshape(-1).view(torch.uint8)
    torch.cuda.synchronize()
    out = []
    for p in (f.data_ptr(), buf.data_ptr() + off):
        with S.Sadi(N, 1.4, 0.9, 0.2 / (N + 1)) as s:
            s.set_options(1, getattr(S, prec_name))
            s.set_initial(WL.gaussian_bumps(N, 4, 4500 + N))
            for _ in range(2):
                s.sadi_step_source(p, dtype)
            out.append(s.get()[0])
    assert np.array_equal(out[0], out[1])
