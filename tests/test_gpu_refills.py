"""Refilled rows in rounds of more than 32 merges: a row that asked is served
once, and its list is taken, also when the round it was scanned in makes up to
63 merges (single linkage takes them one after another along a chain).
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_06816_gb300 import Context  # noqa: E402

BLOCK, BLOCKS, GROUPS = 32, 21, 10


def _chains():
    """Ten chains of 60 objects (three in each of twenty 32-row blocks), one a round,
    16 rows whose nearest columns all lie in the first chain, and 56 objects that
    stay live until the chains are done and are the next nearest of all rows."""
    n = BLOCK * BLOCKS
    slot = np.arange(n)
    block, at = slot // BLOCK, slot % BLOCK
    chain = np.where((block < 20) & (at >= 1) & (at <= 30), (at - 1) // 3, -1)
    asks = (at == 0) & (block < 16)
    late = (chain < 0) & ~asks
    rng = np.random.default_rng(5)
    D = 70.0 + rng.random((n, n))
    small = rng.random((n, n)) * 1e-2
    D[np.ix_(chain >= 0, late)] = 40.0 + small[np.ix_(chain >= 0, late)]
    D[np.ix_(asks, chain >= 1)] = 65.0 + small[np.ix_(asks, chain >= 1)]
    D[np.ix_(asks, late)] = 32.0 + small[np.ix_(asks, late)]
    D[np.ix_(asks, chain == 0)] = 20.0 + small[np.ix_(asks, chain == 0)]
    D = np.minimum(D, D.T)
    for g in list(range(GROUPS)) + [-1, -2]:
        members = slot[late if g == -1 else asks if g == -2 else chain == g]
        base = {-1: 25.0, -2: 31.0}.get(g, 1.0 + g)
        for k, (a, b) in enumerate(zip(members[:-1], members[1:])):
            D[a, b] = D[b, a] = base + 1e-2 * k
    return D[np.triu_indices(n, 1)].astype(np.float32), n


def test_lists_of_long_rounds_are_taken():
    """The 16 rows lose their keys in the first round and ask once; a chain's
    survivor (two at most per round) asks once; when the late objects merge, the
    26 rows left ask again, and the ten survivors after the 16 rows: 16 + 20 + 26 +
    10 served rows, and some whose answer came too late.  Dropping the lists
    of long rounds serves the 16 rows in every round while the chains last (16 * 8)."""
    D, n = _chains()
    want = oracle.cached(D, n, 0)
    ctx = Context(0)
    ctx.set_grid(BLOCKS)
    m, h = ctx.cluster(torch.from_numpy(D).cuda(), n, 0)
    torch.cuda.synchronize()
    st = ctx.stats()
    ctx.close()
    np.testing.assert_array_equal(m.cpu().numpy(), want[0])
    np.testing.assert_array_equal(h.cpu().numpy(), np.asarray(want[1], np.float32))
    assert st["rounds"] <= 40, st  # (else the rounds are not the ones meant)
    assert st["refills"] <= 100, st
    assert st["installs"] <= st["refills"], st
