"""fio_solve with inner = FIO_PTF32X3: which arithmetic its corrections run in.

The operator's butterfly stages have 450 blocks of 128 rows: above two tiles for every multiprocessor, with work
enough for the 30-bit fixed-point kernel at b = 32.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder.pack import pack  # noqa: E402
from paper_2105_02995_gb300.builder.stages import KIND_INPLACE, KIND_MAP, Stage  # noqa: E402

B, X3 = 32, binding.FIO_PTF32X3


@pytest.fixture(scope="module")
def setup():
    fbuild.build()
    rng = np.random.default_rng(9)
    m, N = 128, 128 * 450
    q, _ = np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))

    def stage(inplace, count):  # (in-place blocks of 64 rows: no split kernel, whose sums are in another order)
        st, pin, pout = Stage(KIND_INPLACE if inplace else KIND_MAP, N, N), rng.permutation(N), rng.permutation(N)
        w = 64 if inplace else m
        for k in range(0, w * count, w):
            M = np.eye(w) + 1e-3 * rng.standard_normal((w, w)) if inplace else q * np.exp(2j * np.pi * rng.random((w, 1)))
            st.add(M, pin[k:k + w], (pin if inplace else pout)[k:k + w])
        return st

    op = binding.Operator(pack(1, N, [stage(False, 450) for _ in range(2)], [stage(True, 40)], [stage(True, 1)], 0.0, 0.0))
    u = binding.colmajor(torch.from_numpy(rng.standard_normal((N, B)) + 1j * rng.standard_normal((N, B))).to("cuda"))
    yield op, u
    op.release()


def step(op, u):
    """One correction from a zero guess, G-dot K-dot* u (its residual is above the tolerance)."""
    return op.solve(u, method=binding.FIO_IR, inner=X3, tol=1e-30, maxit=1)[0]


def single(op, u, prec):
    return op.apply_inv(binding.colmajor(u.to(torch.complex64)), precision=prec).to(torch.complex128)


def test_direct_is_the_precision_asked_for(setup):
    op, u = setup
    f, _ = op.solve(u, method=binding.FIO_DIRECT, inner=X3)
    assert torch.equal(f, single(op, u, X3))


def test_corrections_do_not_depend_on_the_fp32_variant(setup):
    op, u = setup
    want = step(op, u)
    try:
        op.set_variant(B, binding.FIO_P32, 3)
        assert torch.equal(step(op, u), want)
    finally:
        op.set_variant(B, binding.FIO_P32, 0)
    op.autotune(B, X3)
    exact = op.apply_inv(u)
    # the fixed-point stages still serve: nearer than tuned split TF32
    near, split = ((v - exact).abs().max() for v in (step(op, u), single(op, u, X3)))
    assert near < split
    op.set_variant(B, X3, 0)


def test_a_pinned_variant_is_used(setup):
    op, u = setup
    try:
        op.set_variant(B, X3, 22)
        assert torch.equal(step(op, u), single(op, u, X3))
    finally:
        op.set_variant(B, X3, 0)
    assert not torch.equal(step(op, u), single(op, u, X3))
