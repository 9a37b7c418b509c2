"""sadi_autotune of the dense form on the shared-memory engine leaves the y-sweep
tile alone: its y sweep is a GEMM, so candidates that differ there are the same
step and only noise could choose between them."""
import pytest

pytestmark = pytest.mark.gpu


def test_autotune_of_the_dense_form_has_no_y_sweep_tile():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_06206_gb300 import build
    build.build()
    from paper_2312_06206_gb300 import sadi as S
    ctxs = [S.Sadi(N, 1.5, 1.0, 0.2 / (N + 1)) for N in (4089, 4090, 4095)]
    for s in ctxs:
        s.set_options(1, S.SADI_PREC_FP32_DENSE)
    default = [s.sadi_get_tiles()[2] for s in ctxs]
    S.sadi_autotune(ctxs, 1, 2)
    assert [s.sadi_get_tiles()[2] for s in ctxs] == default
    for s in ctxs:
        s.close()
