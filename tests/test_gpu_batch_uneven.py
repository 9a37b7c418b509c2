"""Batched steps of members with different N in one FFT length, bitwise against
each member alone: the block-FFT kernels with whole groups of rows (clusters at
N' = 1024 and 2048) that exit early, border ranks on both sides of 32 in one
launch, and dense sweeps with one shared-memory layout per member.

The kernels' decomposition and order of summation do not depend on what else is
in the launch, so the fields are equal bit for bit, in every repetition."""
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


def _make(S, prec_name, members):
    out = []
    for N, kappa in members:
        s = S.Sadi(N, 1.5, kappa, 0.3 / (N + 1))
        s.set_options(1, getattr(S, prec_name))
        s.set_initial(WL.gaussian_bumps(N, 4, 4200 + N), 0.1 * WL.gaussian_bumps(N, 3, 4300 + N))
        out.append(s)
    return out


CASES = {
    # clusters of two blocks: 32 / 33 border columns, none, one, and many
    "gs-1024": ("SADI_PREC_FP32", [(1023, 1.0), (1024, 1.0), (991, 0.7), (992, 1.3), (600, 1.0)]),
    # dense sweeps from r = 33 on (large kappa: H^-1 held whole, else I + E),
    # the transforms' sweeps with the border inline up to r = 32
    "gs-512": ("SADI_PREC_FP32", [(300, 1.0), (400, 900.0), (479, 0.7), (480, 1.0), (511, 1.3)]),
    "gs-256": ("SADI_PREC_FP32", [(129, 900.0), (223, 1.0), (224, 1.0), (255, 0.7), (256, 1.0)]),
    "gs-128": ("SADI_PREC_FP32", [(65, 1.0), (80, 900.0), (95, 0.7), (96, 1.0), (127, 1.3), (128, 1.0)]),
    "dense-1024": ("SADI_PREC_FP32_DENSE", [(1023, 1.0), (600, 1.0), (1024, 0.7)]),
    # clusters of eight
    "dense-2048": ("SADI_PREC_FP32_DENSE", [(2047, 1.0), (2048, 1.0), (2041, 0.7), (1990, 1.3)]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_batch_equals_members_alone(S, name):
    prec_name, members = CASES[name]
    alone = _make(S, prec_name, members)
    batches = [_make(S, prec_name, members) for _ in range(2)]
    for s in alone:
        s.step(4)
    for b in batches:
        S.sadi_batch_step(b, 4)
    for k, s in enumerate(alone):
        u = s.get()[0]
        assert np.isfinite(u).all() and np.abs(u).max() > 0.0
        for b in batches:
            assert np.array_equal(u, b[k].get()[0]), members[k]
    for s in alone + batches[0] + batches[1]:
        s.close()
