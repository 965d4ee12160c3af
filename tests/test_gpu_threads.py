"""Contexts of several threads, each with a matrix of its own size: a kernel's limit of
shared memory belongs to the function, and a thread with a smaller matrix must
not lower it under a launch of another.
"""
import threading

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_06816_gb300 import Context  # noqa: E402


@pytest.mark.parametrize("grid,sizes", [(0, (430, 520, 700, 1500)), (1, (64, 130, 300, 420))])
def test_threads_with_matrices_of_different_sizes(grid, sizes):
    passes, errors = 200, []
    start = threading.Barrier(len(sizes), timeout=60)

    def work(n):
        try:
            D = synth.small_gmm(n, n, dim=6, k=5)
            want_m, want_h, _, _ = oracle.cached(D, n, 1)
            stream = torch.cuda.Stream()
            ctx = Context(0, stream=stream)
            ctx.set_grid(grid)
            with torch.cuda.stream(stream):
                src = torch.from_numpy(D).cuda()
                buf = torch.empty_like(src)
                start.wait()
                for _ in range(passes):
                    buf.copy_(src)
                    m, h = ctx.cluster(buf, n, 1)
                stream.synchronize()
            ctx.close()
            np.testing.assert_array_equal(m.cpu().numpy(), want_m)
            np.testing.assert_array_equal(h.cpu().numpy().view(np.uint32),
                                          np.asarray(want_h, np.float32).view(np.uint32))
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append((n, repr(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
