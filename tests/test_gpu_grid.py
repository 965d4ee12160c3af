"""The automatic grid where the number of 32-row blocks is odd: no CTA owns more
blocks than two when one CTA per two blocks fits the device.
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


@pytest.mark.parametrize("n", [4096, 4097, 4128, 4129, 5003])
def test_odd_block_counts(n):
    D = synth.small_gmm(n, 80, dim=6, k=5)
    ctx = Context(0)
    m, h = ctx.cluster(torch.from_numpy(D).cuda(), n, 2)
    torch.cuda.synchronize()
    grid = ctx.stats()["grid"]
    ctx.close()
    blocks = (n + 31) // 32
    assert -(-blocks // grid) == 2
    want_m, want_h, _, _ = oracle.cached(D, n, 2)
    np.testing.assert_array_equal(m.cpu().numpy(), want_m)
    np.testing.assert_array_equal(h.cpu().numpy().view(np.uint32), np.asarray(want_h, np.float32).view(np.uint32))
