"""Fixed-point stages over the range of their operands: vectors near the lower end of the exponents.

Tolerance: the bound of test_gpu_fixed_point (its operator has the same number of stages, of the same
growth): 1.8e-14 of the result in the measure of the largest and of the 2-norm.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import factor_apply as fa  # noqa: E402
from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder.pack import pack  # noqa: E402
from paper_2105_02995_gb300.builder.stages import KIND_INPLACE, KIND_MAP, Stage  # noqa: E402

TOL64 = 1.8e-14
REFS = {"K": fa.apply_Kdot, "Kadj": fa.apply_Kdot_adj, "G": fa.apply_G, "inv": fa.apply_inv}
SIDES = [7, 16, 33, 64, 130, 260] + [58] * 90
_ops = {}


def gaussian(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def operator(kind, map_block, hif_block, sides=SIDES):
    """Three butterfly stages and a HIF level of ragged blocks above 4096 unknowns, where every FP64
    stage takes the kernel from five right-hand sides on."""
    if kind not in _ops:
        fbuild.build()
        rng = np.random.default_rng(7)
        N = sum(sides)

        def stage(inplace):
            st, i = Stage(KIND_INPLACE if inplace else KIND_MAP, N, N), 0
            pin, pout = rng.permutation(N), rng.permutation(N)
            for m in rng.permutation(sides):
                rows = pin if inplace else pout
                st.add((hif_block if inplace else map_block)(rng, m), pin[i:i + m], rows[i:i + m])
                i += m
            return st

        buf = pack(1, N, [stage(False) for _ in range(3)], [stage(True)], [stage(True)], 0.0, 0.0)
        _ops[kind] = (binding.Operator(buf), fa.PackedFactors(buf), N)
    return _ops[kind]


def even(rng, m):
    return gaussian(rng, m, m) / (2 * np.sqrt(m))


def near_identity(rng, m):
    return np.eye(m) + 0.1 * even(rng, m)


def dev(a, dtype=torch.complex128):
    return binding.colmajor(torch.from_numpy(np.asarray(a)).to("cuda", dtype))


def rel(a, b):
    return max(float(np.linalg.norm(a - b) / np.linalg.norm(b)), float(np.abs(a - b).max() / np.abs(b).max()))


@pytest.mark.parametrize("k", [940, 965, 975, 981, 990])
def test_zeros_in_tiny_columns(k):
    """Zeros, and the zero imaginary parts of a real right-hand side, are zeros at every scale."""
    op, P, N = operator("even", even, near_identity)
    x = np.random.default_rng(k).standard_normal((N, 9)) + 0j
    x[::3] = 0.0
    for w, ref in REFS.items():
        y = getattr(op, "apply_" + w)(dev(x * 2.0 ** -k)).cpu().numpy() * 2.0 ** k
        assert rel(y, ref(P, x)) < TOL64, w


def graded(rng, m):
    """Rows and columns that span 20 binary orders each."""
    return np.exp2(rng.uniform(-20, 0, (m, 1))) * even(rng, m) * np.exp2(rng.uniform(-20, 0, (1, m)))


def hermitian(rng, m):
    """A scaled positive definite block, as HIF and root blocks are: diagonal 2^-16 .. 1."""
    e, d = even(rng, m), np.exp2(rng.uniform(-8, 0, m))
    return d[:, None] * (np.eye(m) + 0.2 * (e + e.conj().T)) * d


def wide(S, x, adjoint):
    """A stage's product in extended precision."""
    return (S.conj().T if adjoint else S).tocsr().astype(np.clongdouble) @ x.astype(np.clongdouble)


BLOCKS = {"even": (even, near_identity), "graded": (graded, hermitian), "hermitian": (hermitian, graded)}


@pytest.mark.parametrize("vector", ["gaussian", "40 orders", "against the factor", "half against"])
@pytest.mark.parametrize("kind", list(BLOCKS))
def test_error_no_larger_than_an_fma_chain(kind, vector):
    """Factors and vectors whose entries span many binary orders, large entries of the one meeting small
    ones of the other: no further from the product in extended precision than the CUDA-core sums."""
    op, P, N = operator(kind, *BLOCKS[kind])
    b = 6
    rng = np.random.default_rng(41)
    for w, S, adjoint in (("K", P.bf[0], False), ("Kadj", P.bf[2], True), ("G", P.hif[0], False)):
        x = gaussian(rng, N, b)
        cols = abs(S.conj().T if adjoint else S).max(axis=0).toarray().ravel()[:, None]
        x = {"gaussian": x, "40 orders": x * np.exp2(rng.uniform(-40, 0, (N, 1))), "against the factor": x / cols,
             "half against": x / np.sqrt(cols)}[vector]
        chain = {"K": [(s, False) for s in P.bf], "Kadj": [(s, True) for s in reversed(P.bf)],
                 "G": [(P.hif[0], False), (P.root[0], False), (P.hif[0], True)]}[w]
        want = x
        for s, a in chain:
            want = wide(s, want, a)
        xd, fn = dev(x), getattr(op, "apply_" + w)
        y = fn(xd).cpu().numpy()
        try:
            op.set_variant(b, binding.FIO_P64, 1)
            z = fn(xd).cpu().numpy()
        finally:
            op.set_variant(b, binding.FIO_P64, 0)
        assert not np.array_equal(y, z)  # the two kernels
        ey, ez = (float(np.sqrt((np.abs(v - want) ** 2).sum() / (np.abs(want) ** 2).sum())) for v in (y, z))
        assert ey <= ez, (w, ey, ez)


@pytest.mark.parametrize("b", [1, 8, 9, 16, 17, 32, 33])
@pytest.mark.parametrize("prec", [binding.FIO_P64, binding.FIO_P32])
def test_short_blocks(prec, b):
    """Stages whose gathers keep all of a thread's entries (blocks of at most 58 columns), some of one column.
    FP32: 2 2^-24 a stage, as in test_gpu_fixed_point."""
    op, P, N = operator("short", even, near_identity, [1, 2, 33, 57] + [58] * 110)
    wide = prec == binding.FIO_P64
    xd = dev(gaussian(np.random.default_rng(b), N, b), torch.complex128 if wide else torch.complex64)
    x = xd.cpu().numpy().astype(np.complex128)
    try:
        op.set_variant(b, prec, 50)
        for w in ("K", "Kadj"):
            y = getattr(op, "apply_" + w)(xd, precision=prec).cpu().numpy().astype(np.complex128)
            assert rel(y, REFS[w](P, x)) < (TOL64 if wide else 1.1e-6), w
    finally:
        op.set_variant(b, prec, 0)
