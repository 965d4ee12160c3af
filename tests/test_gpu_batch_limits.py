"""A class of one-CTA batch jobs whose limit lies above what a CTA of its size
holds (the shipped table ends at 4096): the jobs in between run over the device.
"""
import json
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_06816_gb300 as pkg  # noqa: E402

TUNED = os.path.join(os.path.dirname(pkg.__file__), "tuned", "batch_NVIDIA_GB300_152.json")


def _shipped():
    with open(TUNED) as f:
        return [tuple(c) for c in json.load(f)["classes"]]


@pytest.mark.parametrize("classes", [None, [(4096, 128)], [(4096, 256)], [(3800, 256), (4096, 512)]])
def test_jobs_above_what_one_cta_holds(classes):
    ctx = pkg.Context(0)
    ctx.set_batch_classes(_shipped() if classes is None else classes)
    sizes = [64, 3200, 3521, 3800, 4096, 4097]
    data = [synth.small_gmm(n, 70 + q, dim=6, k=5) for q, n in enumerate(sizes)]
    mats = [torch.from_numpy(D).cuda() for D in data]
    outs, status = ctx.cluster_batch(mats, sizes, [1] * len(sizes))
    torch.cuda.synchronize()
    ctx.close()
    assert list(status) == [0] * len(sizes)
    for (m, h), D, n in zip(outs, data, sizes):
        want_m, want_h, _, _ = oracle.cached(D, n, 1)
        np.testing.assert_array_equal(m.cpu().numpy(), want_m)
        np.testing.assert_array_equal(h.cpu().numpy().view(np.uint32), np.asarray(want_h, np.float32).view(np.uint32))
