"""The survivors' lists when far more new cells than they hold lie below their
limit (equal values): the smallest stay listed, so that the next round has
entries of that row and not a bare mark.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_06816_gb300 import Context  # noqa: E402


def _values(kind, n):
    rng = np.random.default_rng(n)
    cells = n * (n - 1) // 2
    if kind == "one":
        return np.full(cells, 1.25, np.float32)
    if kind == "levels":
        return rng.integers(1, 5, cells).astype(np.float32)
    # columns 64 apart share a place: every row's small cells lie there
    c = np.broadcast_to(np.arange(n), (n, n))[np.triu_indices(n, 1)]
    return (rng.random(cells) + np.where(c % 64 == 7, 1.0, 3.0)).astype(np.float32)


@pytest.mark.parametrize("kind", ["one", "levels", "columns"])
@pytest.mark.parametrize("link", range(6))
@pytest.mark.parametrize("grid,layout", [(0, 0), (3, 2)])
def test_lists_that_run_over(kind, link, grid, layout):
    n = 900
    D = _values(kind, n)
    want = oracle.cached(D, n, link)
    ctx = Context(0)
    ctx.set_grid(grid or 29)
    ctx.set_layout(layout)
    m, h = ctx.cluster(torch.from_numpy(D).cuda(), n, link)
    torch.cuda.synchronize()
    ctx.close()
    np.testing.assert_array_equal(m.cpu().numpy(), want[0])
    np.testing.assert_array_equal(h.cpu().numpy().view(np.uint32), np.asarray(want[1], np.float32).view(np.uint32))


@pytest.mark.parametrize("link", [0, 3])
def test_one_value_leaves_no_idle_rounds(link):
    """One value everywhere: every survivor's row ties.  Lists in order of arrival
    left every second to fourth round without a merge."""
    n = 2000
    ctx = Context(0)
    ctx.cluster(torch.full((n * (n - 1) // 2,), 1.25, device="cuda"), n, link)
    st = ctx.stats()
    ctx.close()
    assert 16 * st["idle_rounds"] <= st["rounds"], st
