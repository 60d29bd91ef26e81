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


def operator(kind, map_block, hif_block):
    """Three butterfly stages and a HIF level of ragged blocks above 4096 unknowns, where every FP64
    stage takes the kernel from five right-hand sides on."""
    if kind not in _ops:
        fbuild.build()
        rng = np.random.default_rng(7)
        N = sum(SIDES)

        def stage(inplace):
            st, i = Stage(KIND_INPLACE if inplace else KIND_MAP, N, N), 0
            pin, pout = rng.permutation(N), rng.permutation(N)
            for m in rng.permutation(SIDES):
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
