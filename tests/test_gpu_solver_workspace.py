"""The solvers do not depend on what lies in their work arrays when these are allocated."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder import build_operator  # noqa: E402


@pytest.fixture(scope="module")
def packed():
    fbuild.build()
    return build_operator("ex1", 1024, 1e-7, 1e-6)[0]


@pytest.mark.parametrize("b", [1, 5])
@pytest.mark.parametrize("method", [binding.FIO_PCG, binding.FIO_GMRES, binding.FIO_IR, binding.FIO_DIRECT])
def test_nan_in_the_work_arrays(packed, method, b):
    op = binding.Operator(packed)
    u = binding.colmajor(torch.randn((1024, b), dtype=torch.complex128, device="cuda"))
    torch.cuda.synchronize()
    # NaN in what the driver hands out next: the operator's own scratch, freed each time it grows
    for k in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 128):
        op.apply_inv(binding.colmajor(torch.full((1024, k), float("nan"), dtype=torch.complex128, device="cuda")))
    torch.cuda.synchronize()
    f, info = op.solve(u, method=method, tol=1e-10, maxit=40)
    assert bool(torch.isfinite(torch.view_as_real(f)).all())
    assert all(s == 0 for _, _, s in info), info
    op.release()
