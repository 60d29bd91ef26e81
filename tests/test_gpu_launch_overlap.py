"""Stage launches that are started early lose no time.

Butterfly stages of 16 x 16 and of 230 x 230 blocks in FP64: five and eight right-hand sides run the same
tiles of eight columns, as long as one another.  Where the narrower tile counted as light and its launches
were started ahead, its CTAs shared multiprocessors and K-dot took 1.7 times as long.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2105_02995_gb300 import binding, build as fbuild  # noqa: E402
from paper_2105_02995_gb300.builder.pack import pack  # noqa: E402
from paper_2105_02995_gb300.builder.stages import KIND_MAP, Stage  # noqa: E402


def test_narrow_batches_of_heavy_tiles():
    fbuild.build()
    rng = np.random.default_rng(5)
    N = 230 * 10

    def stage(width):
        st, pin, pout = Stage(KIND_MAP, N, N), rng.permutation(N), rng.permutation(N)
        for k in range(0, N, width):
            m = min(width, N - k)
            st.add(rng.standard_normal((m, m)) / np.sqrt(m) + 0j, pin[k:k + m], pout[k:k + m])
        return st

    op = binding.Operator(pack(1, N, [stage(16)] + [stage(230) for _ in range(4)], [], [], 0.0, 0.0))
    best = {}
    for _ in range(5):
        for b in (5, 8):
            x = torch.ones((b, N), dtype=torch.complex128, device="cuda").t()
            y = binding.colmajor(torch.empty_like(x))
            op.apply_K(x, y)
            t0, t1 = torch.cuda.Event(True), torch.cuda.Event(True)
            t0.record()
            for _ in range(8):
                op.apply_K(x, y)
            t1.record()
            torch.cuda.synchronize()
            best[b] = min(best.get(b, 1e9), t0.elapsed_time(t1))
    assert best[5] < 1.25 * best[8], best
    op.release()
