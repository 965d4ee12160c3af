"""Rounds of the merge kernel at the sizes and values where their parts can go
wrong: the default grid on both sides of each of its lines, CTAs with more rows
than a publish pass holds heads for, merges taken on condition and put off
again (ties), lists of new cells that run over (one value everywhere), bounds
without a relative margin (zeros, the smallest and very large values).  Every
result is the oracle's, bit for bit.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_06816_gb300 import Context  # noqa: E402


def _values(kind, n, seed):
    cells = n * (n - 1) // 2
    if kind == "gmm":
        return synth.small_gmm(n, seed)
    if kind == "ties":
        return synth.tie_heavy(n, seed, levels=3)
    if kind == "one":
        return np.full(cells, 1.25, dtype=np.float32)
    rng = np.random.default_rng(seed)
    if kind == "zeros":  # half of the cells
        return (rng.random(cells, dtype=np.float32) * (rng.random(cells) < 0.5)).astype(np.float32)
    return (rng.random(cells) + 0.5).astype(np.float32) * np.float32({"tiny": 2e-38, "large": 5e36}[kind])


CASES = [(n, link, "gmm", 0, 0, 0) for n in (416, 417, 1152, 1153) for link in (0, 3, 5)]
CASES += [(2080, 1, "gmm", 0, 0, 0), (2080, 2, "ties", 0, 0, 0)]
CASES += [(610, link, kind, 0, grid, layout) for link in range(6)
          for kind, grid, layout in (("ties", 0, 0), ("one", 5, 2), ("zeros", 1, 0), ("zeros", 19, 1),
                                     ("tiny", 0, 0), ("large", 0, 0))]
CASES += [(1300, 1, "gmm", 128, 2, 1), (1300, 2, "ties", 128, 2, 2), (1300, 4, "ties", 256, 1, 0)]


@pytest.mark.parametrize("n,link,kind,nt,grid,layout", CASES)
def test_rounds(n, link, kind, nt, grid, layout):
    D = _values(kind, n, n + link)
    want = oracle.cached(D, n, link)
    ctx = Context(0)
    ctx.set_grid(grid)
    ctx.set_layout(layout)
    ctx.set_cta_threads(nt)
    m, h = ctx.cluster(torch.from_numpy(D).cuda(), n, link)
    torch.cuda.synchronize()
    ctx.close()
    np.testing.assert_array_equal(m.cpu().numpy(), want[0])
    np.testing.assert_array_equal(h.cpu().numpy().view(np.uint32), np.asarray(want[1], np.float32).view(np.uint32))
