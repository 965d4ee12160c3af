"""Ward linkage on values whose recurrence overflows FP32: cells become infinite,
and NaN when an infinite one is merged (0 * inf in the last term).  Neither is
refused: they order behind every number, as in the oracle, so the merges stay the
oracle's to the end.  Heights are its bits up to the first NaN; a NaN has no
bits of its own (host and device differ).
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_06816_gb300 import Context  # noqa: E402


# one CTA (a warp scans a row), grids on the packed triangle (a CTA scans a row)
# and on the row-log layout
@pytest.mark.parametrize("n,grid,layout", [(100, 1, 0), (400, 1, 0), (1100, 1, 0), (400, 3, 2), (1500, 5, 2),
                                           (1500, 0, 2), (1500, 0, 1)])
def test_overflowing_ward(n, grid, layout):
    rng = np.random.default_rng(n)
    D = (rng.random(n * (n - 1) // 2) * 3.4e38).astype(np.float32)
    want_m, want_h = oracle.cached(D, n, 3)[:2]
    want_h = np.asarray(want_h, np.float32)
    ctx = Context(0)
    ctx.set_grid(grid)
    ctx.set_layout(layout)
    m, h = ctx.cluster(torch.from_numpy(D).cuda(), n, 3)
    torch.cuda.synchronize()
    ctx.close()
    m, h = m.cpu().numpy(), h.cpu().numpy()
    assert np.isinf(want_h).any() and np.isnan(want_h).any()
    np.testing.assert_array_equal(m, want_m)
    np.testing.assert_array_equal(np.isnan(h), np.isnan(want_h))
    number = ~np.isnan(want_h)
    np.testing.assert_array_equal(h[number].view(np.uint32), want_h[number].view(np.uint32))
