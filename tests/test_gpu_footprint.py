"""Device memory of a context at N' = 8192: the arrays that its steps and its
set-up read, and no table of a path that this length does not take."""
import pytest

pytestmark = pytest.mark.gpu


def test_context_holds_no_unread_tables():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_06206_gb300 import build
    build.build()
    from paper_2312_06206_gb300 import sadi as S
    N, Np = 8190, 8192
    S.Sadi(63, 1.5, 1.0, 1e-3).close()         # the library's own first allocations
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = S.Sadi(N, 1.5, 1.0, 1e-4)
    grown = before - torch.cuda.mem_get_info()[0]
    s.close()
    doubles = (N * N                            # weights a_ij
               + (Np + 1) ** 2                  # symbol
               + 3 * (Np + 1) * Np              # its rows for the engine, FP64 and FP32
               + N * N                          # staging
               + 4 * N * N                      # state, phi2, sweep scratch
               + 2 * N * Np)                    # spectrum
    # vectors of N' entries and the 2 MB granularity of large allocations
    assert grown <= 8 * doubles + (96 << 20), grown
