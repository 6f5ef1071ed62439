"""The quasar draw's bound on P and its accept bits at the edges: boxes smaller
than a sub-range, densities at which many voxels pass the bound or P reaches 1,
wide fields, both strides."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_qso_draw import compare, params, records

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


@pytest.mark.parametrize("n,nbar,scale,stride", [(2, 0.05, 1.0, 1), (8, 0.02, 0.7, 1), (16, 0.3, 1.5, 2),
                                                 (32, 2e-5, 3.0, 1), (32, 1e-3, 0.0, 2)])
def test_bound_keeps_every_decision(n, nbar, scale, stride):
    c = mk.Context(0)
    q = params(n, 2.19, seed=0xABC0 + n, nbar=nbar)
    rng = np.random.default_rng(n)
    boxes = [(rng.standard_normal((n, n, n)) * scale * s).astype(np.float32) for s in (1.0, 0.8, 0.9)]
    dev = [torch.from_numpy(b.ravel()).cuda() for b in boxes]
    if stride == 2:
        dev = [torch.stack([b, b + 7.0], 1).reshape(-1).contiguous() for b in dev]
    cat, cnt = c.draw_qso(q, dev, stride=stride, capacity=n ** 3)
    ids, pos = records(cat)
    ref = oracle.qso_draw(q, boxes)
    assert cnt == ids.size
    nd = compare(ids, pos, ref, rel=1e-5)
    assert abs(cnt - ref["count"]) <= nd <= 2
    c.close()
