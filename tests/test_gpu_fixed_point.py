"""The fixed-point tensor-core stage kernel (FP64 and FP32 stage products as exact sums of 8-bit
digit products) against the oracle's FP64 product of the same factors.

The operator is random, of about 10,000 unknowns (above the size at which every FP64 stage takes the
kernel; in FP32 it is pinned) in ragged blocks whose sides lie on both sides of the kernel's tiles: 8-column K steps and
their halves, 16-column FP32 chunks, 32-row copies, 128-row tiles, 128- and 256-column drains.

Tolerances.  A stage's outputs are sums without rounding of operands cut to 2^-62 (FP64) resp. 2^-30
(FP32) of their row's and column's largest, rounded once: u = 2^-53 resp. 2^-24 per stage, in the
measure max|a - b| / max|b| at most (stages) u (1 + growth) with unit-norm stages.  The oracle's own
FP64 sums of up to 300 terms add sqrt(300) 2^-53 per stage.  Over the 3 stages of K-dot and the 9
launches of G-dot K-dot*: 9 (1 + 17) 2^-53 = 1.8e-14 and 9 * 2 * 2^-24 = 1.1e-6.
"""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import factor_apply as fa  # noqa: E402
from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder.pack import pack  # noqa: E402
from paper_2105_02995_gb300.builder.stages import KIND_INPLACE, KIND_MAP, Stage  # noqa: E402

FIXED_POINT = 50
TOL = {binding.FIO_P64: 1.8e-14, binding.FIO_PDF: 1.8e-14, binding.FIO_P32: 1.1e-6}
DTYPE = {binding.FIO_P64: torch.complex128, binding.FIO_PDF: torch.complex128, binding.FIO_P32: torch.complex64}
EDGES = [1, 3, 4, 7, 8, 9, 15, 16, 17, 24, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 255, 256, 257, 300]
REFS = {"K": fa.apply_Kdot, "Kadj": fa.apply_Kdot_adj, "G": fa.apply_G, "inv": fa.apply_inv}
_ops = {}


def random_block(rng, m, n, integer):
    if integer:
        return rng.integers(-1, 2, (m, n)) + 1j * rng.integers(-1, 2, (m, n))
    z = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
    return z * np.exp2(rng.integers(-3, 4, (m, 1))) / (2 * np.sqrt(max(m, n)))  # rows of other scales


def operator(kind):
    if kind in _ops:
        return _ops[kind]
    fbuild.build()
    rng = np.random.default_rng(11)
    integer = kind == "integer"
    sides = EDGES + EDGES[:-1] + [200] * 14 + [64] * 30  # 95 blocks ...
    sides += [40] * 37                                     # ... and enough 128-row tiles for the FP32 copy
    N = sum(sides)

    def map_stage():
        st = Stage(KIND_MAP, N, N)
        rows, cols = rng.permutation(sides), rng.permutation(sides)
        pin, pout, i, o = rng.permutation(N), rng.permutation(N), 0, 0
        for m, n in zip(rows, cols):
            M = random_block(rng, m, n, integer)
            if integer:  # two entries a row at most, so that sums stay small integers
                M[:, 2:] = 0
            st.add(M, pin[i:i + n], pout[o:o + m])
            i, o = i + n, o + m
        return st

    def inplace_stage(widths):
        st = Stage(KIND_INPLACE, N, N)
        p, at = rng.permutation(N), 0
        for w in widths:
            M = np.eye(w) if integer else np.eye(w) + 0.1 * random_block(rng, w, w, False)
            st.add(M, p[at:at + w], p[at:at + w])
            at += w
        return st

    hif = [inplace_stage([256] * 10 + [60] * 9), inplace_stage([28] * 7), inplace_stage([1, 5, 130])]
    buf = pack(1, N, [map_stage() for _ in range(3)], hif, [inplace_stage([333])], 0.0, 0.0)
    _ops[kind] = (binding.Operator(buf), fa.PackedFactors(buf), N)
    return _ops[kind]


def vectors(N, b, seed, integer=False):
    rng = np.random.default_rng(seed)
    if integer:
        return rng.integers(-1, 2, (N, b)) + 1j * rng.integers(-1, 2, (N, b))
    return rng.standard_normal((N, b)) + 1j * rng.standard_normal((N, b))


def dev(a, dtype):
    return binding.colmajor(torch.from_numpy(np.asarray(a)).to("cuda", dtype))


def rel(a, b):
    return max(float(np.linalg.norm(a - b) / np.linalg.norm(b)), float(np.abs(a - b).max() / np.abs(b).max()))


@pytest.mark.parametrize("prec", list(TOL))
@pytest.mark.parametrize("b", [1, 2, 5, 8, 9, 16, 17, 31, 33, 70])
def test_random_operator_vs_oracle(prec, b):
    """Every apply of the kernel's stages within the derived bound; in FP64 the kernel runs on every stage from b = 5 on
    (its rounding differs from the CUDA-core tiles'), and double-float goes the same way."""
    op, P, N = operator("random")
    x = vectors(N, b, 100 + b)
    xd = dev(x, DTYPE[prec])
    x64 = xd.cpu().numpy().astype(np.complex128)
    if prec == binding.FIO_P32:
        op.set_variant(b, prec, FIXED_POINT)
    # (the in-place stages have too few tiles for an FP32 copy: G-dot runs on the CUDA cores there)
    for w in ("K", "Kadj") if prec == binding.FIO_P32 else REFS:
        ref = REFS[w]
        y = getattr(op, "apply_" + w)(xd, precision=prec)
        op.sync()
        assert rel(y.cpu().numpy().astype(np.complex128), ref(P, x64)) < TOL[prec], w
    if prec != binding.FIO_P32 and b >= 5:
        y = op.apply_K(xd, precision=prec)
        try:
            op.set_variant(b, binding.FIO_P64, 1)
            assert not torch.equal(y, op.apply_K(xd, precision=binding.FIO_P64))
        finally:
            op.set_variant(b, binding.FIO_P64, 0)
        op.set_variant(b, binding.FIO_P64, FIXED_POINT)
        assert torch.equal(y, op.apply_K(xd, precision=binding.FIO_P64))
        op.set_variant(b, binding.FIO_P64, 0)


@pytest.mark.parametrize("prec", [binding.FIO_P64, binding.FIO_P32])
@pytest.mark.parametrize("b", [3, 16, 40])
def test_integers_are_exact(prec, b):
    op, P, N = operator("integer")
    x = vectors(N, b, 200 + b, integer=True)
    xd = dev(x, DTYPE[prec])
    op.set_variant(b, prec, FIXED_POINT)
    for w, ref in REFS.items():
        y = getattr(op, "apply_" + w)(xd, precision=prec).cpu().numpy().astype(np.complex128)
        assert np.array_equal(y, ref(P, x)), w


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e307, 1e-307, 5e-324, 0.0])
def test_columns_beyond_the_fixed_point(value):
    """Infinities, NaN and exponents at the ends of the range: the same infinities and NaN, in the
    same places, and the same finite values as the CUDA-core kernels; the other columns unchanged."""
    op, P, N = operator("random")
    b = 9
    x = vectors(N, b, 300)
    with np.errstate(all="ignore"):
        x[:, 4] = x[:, 4] * value if value in (1e307, 1e-307, 5e-324, 0.0) else x[:, 4]
    if not np.isfinite(value):
        x[777, 4] = complex(value, 1.0)
    xd = dev(x, torch.complex128)
    plain = dev(vectors(N, b, 300), torch.complex128)
    for w in ("K", "Kadj", "G"):
        fn = getattr(op, "apply_" + w)
        y = fn(xd).cpu().numpy()
        clean = fn(plain).cpu().numpy()
        op.sync()
        try:
            op.set_variant(b, binding.FIO_P64, 1)
            z = fn(xd).cpu().numpy()
        finally:
            op.set_variant(b, binding.FIO_P64, 0)
        keep = [j for j in range(b) if j != 4]
        assert np.array_equal(y[:, keep], clean[:, keep]), w
        for u, v in ((y[:, 4].real, z[:, 4].real), (y[:, 4].imag, z[:, 4].imag)):
            assert np.array_equal(np.isnan(u), np.isnan(v)) and np.array_equal(np.isinf(u), np.isinf(v)), w
            ok = np.isfinite(v)
            scale = np.abs(v[ok]).max(initial=0.0)
            assert np.all(np.abs(u[ok] - v[ok]) <= TOL[binding.FIO_P64] * scale + 1e-322), w


@pytest.mark.parametrize("prec", [binding.FIO_P64, binding.FIO_P32])
def test_other_entries_agree_bit_for_bit(prec):
    """ld > N, the host-buffer and allocation-free entries and a captured graph: the same kernels."""
    op, P, N = operator("random")
    b = 21
    op.set_variant(b, prec, FIXED_POINT)
    x = dev(vectors(N, b, 400), DTYPE[prec])
    want = op.apply_inv(x, precision=prec)
    big = torch.zeros((b, N + 9), dtype=DTYPE[prec], device="cuda")
    big[:, :N] = x.t()
    out = torch.full_like(big, 7.0)
    op.apply_inv(big.t()[:N], out.t()[:N], precision=prec)
    assert torch.equal(out.t()[:N], want) and torch.all(out[:, N:] == 7.0)
    assert np.array_equal(op.apply_inv_host(np.asfortranarray(x.cpu().numpy()), precision=prec), want.cpu().numpy())
    f = binding.colmajor(torch.empty_like(x))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = binding.load().fio_apply_inv_noalloc(op.h, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(f.data_ptr()), N, b,
                                              binding.FIO_C128 if prec == binding.FIO_P64 else binding.FIO_C64, prec, stream)
    torch.cuda.synchronize()
    assert rc == 0 and torch.equal(f, want)
    g = op.capture_inv(x, f, prec)
    f.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(f, want)
