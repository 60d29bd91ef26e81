"""FIO_PDF on operators whose stages all run in FP64 fixed point: its choices and its diagnostics are its own."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2105_02995_gb300 import binding  # noqa: E402
from test_gpu_fixed_point_range import dev, even, gaussian, near_identity, operator  # noqa: E402


@pytest.mark.parametrize("b", [2, 12])
def test_choices_are_kept_apart(b):
    import numpy as np

    op, _, N = operator("even", even, near_identity)
    x = dev(gaussian(np.random.default_rng(6), N, b))
    df = op.apply_K(x, precision=binding.FIO_PDF)
    try:
        op.set_variant(b, binding.FIO_P64, 1)
        cores = op.apply_K(x)
        assert torch.equal(op.apply_K(x, precision=binding.FIO_PDF), df)
        assert len(op.autotune(b, binding.FIO_PDF)) == 3 * 2 + 1 * 2 + 1
        assert torch.equal(op.apply_K(x), cores)  # the pinned FP64 variant
        if b > 4:
            assert torch.equal(op.apply_K(x, precision=binding.FIO_PDF), df)
    finally:
        op.set_variant(b, binding.FIO_P64, 0)
        op.set_variant(b, binding.FIO_PDF, 0)
    assert torch.equal(op.apply_K(x, precision=binding.FIO_PDF), df)


def test_stage_errors_measure_the_kernel():
    import numpy as np

    op, _, N = operator("even", even, near_identity)
    errs = op.stage_errors("inv", dev(gaussian(np.random.default_rng(8), N, 8)), binding.FIO_PDF)
    # 3 butterfly stages, 2 in-place levels each way around a root: sums of up to 260 terms in FP64
    assert len(errs) == 6 and all(0.0 < e < 6 * (1 + 2 * 17) * 2.0 ** -53 for e in errs), errs
