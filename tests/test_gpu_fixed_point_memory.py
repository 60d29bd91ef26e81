"""What the fixed-point stages hold in device memory, and what they do where it is short.

The operator has two butterfly stages of 450 blocks of 128 x 128 (no padding): 8 bytes an entry in
complex64, and per direction 16 (FP64) and 8 (FP32) in digits.
"""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder.pack import pack  # noqa: E402
from paper_2105_02995_gb300.builder.stages import KIND_MAP, Stage  # noqa: E402

M, BLOCKS, STAGES = 128, 450, 2
N, ENTRIES = M * BLOCKS, STAGES * BLOCKS * M * M
DIGITS64, DIGITS32 = 2 * 16 * ENTRIES, 2 * 8 * ENTRIES


@pytest.fixture(scope="module")
def packed():
    fbuild.build()
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M)))

    def stage():
        st, pin, pout = Stage(KIND_MAP, N, N), rng.permutation(N), rng.permutation(N)
        for k in range(0, N, M):
            st.add(q * np.exp(2j * np.pi * rng.random((M, 1))), pin[k:k + M], pout[k:k + M])
        return st

    return pack(1, N, [stage() for _ in range(STAGES)], [], [], 0.0, 0.0)


def held(op):
    nb = ctypes.c_size_t()
    assert binding.load().fio_query(op.h, None, None, None, ctypes.byref(nb)) == 0
    return nb.value


def vectors(b, dtype, seed=1):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn((b, N), dtype=torch.complex128, device="cuda", generator=g).to(dtype).t()


class Hog:
    """Takes device memory until `leave` bytes are free."""

    def __init__(self, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.t = [torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")]

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.t.clear()
        torch.cuda.empty_cache()


def test_fp32_copies_are_made_for_tensor_core_operators_only(packed):
    """Plain FP32 applies never reach them, and take no scratch for them."""
    ops = [binding.Operator(packed, m) for m in (binding.FIO_MASK_P64, binding.FIO_MASK_P64 | binding.FIO_MASK_P32)]
    assert held(ops[1]) - held(ops[0]) < 8 * ENTRIES + (1 << 20)
    before, b = held(ops[1]), 32
    ops[1].apply_K(vectors(b, torch.complex64), precision=binding.FIO_P32)
    assert held(ops[1]) - before <= 5 * (8 * N * b + 256)
    for op in ops:
        op.release()


def test_fp64_copies_come_first(packed):
    """Where only FP64's digit copies fit half of the free memory, they are made."""
    x = vectors(8, torch.complex128)
    full = binding.Operator(packed)
    want, arenas = full.apply_K(x), held(full) - DIGITS64 - DIGITS32
    full.release()
    with Hog(arenas + 2 * DIGITS64 + DIGITS32):
        op = binding.Operator(packed)
    assert held(op) < arenas + DIGITS64 + DIGITS32 // 2
    assert torch.equal(op.apply_K(x), want)
    op.release()


def test_scratch_that_does_not_fit_is_asked_for_again(packed):
    """One call without room for the fixed-point scratch runs on the CUDA cores; the calls after it do not."""
    op, wide = binding.Operator(packed), 96
    x8, x = vectors(8, torch.complex128), vectors(wide, torch.complex128)
    want8, out = op.apply_K(x8), binding.colmajor(torch.empty_like(x))
    op.set_variant(wide, binding.FIO_P64, 1)
    cores = op.apply_K(x)
    op.set_variant(wide, binding.FIO_P64, 0)
    op.release()
    op = binding.Operator(packed)
    torch.cuda.Stream()  # torch's streams are made before memory is short
    pool = 5 * 16 * N * wide  # and 1/5 of it for the fixed-point kernel
    with Hog(pool + pool // 10):
        op.apply_K(x, out)
        torch.cuda.synchronize()
        assert held(op) >= pool
        assert torch.equal(out, cores)
        graph = torch.cuda.CUDAGraph()  # a captured call allocates nothing either
        with torch.cuda.graph(graph):
            op.apply_K(x, out)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
    assert torch.equal(out, cores)
    assert torch.equal(op.apply_K(x8), want8)
    assert not torch.equal(op.apply_K(x, out), cores)
    op.release()
