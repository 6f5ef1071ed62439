"""The quasar draw gives large device scratch back, and draws the same afterwards."""
import pytest

from tests.test_gpu_qso_draw import params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


def test_scratch_of_a_large_draw_is_given_back():
    n = 2048
    c = mk.Context(0)
    small = [torch.zeros(64 ** 3, device="cuda")] * 3
    c.draw_qso(params(64, 2.19, seed=1), small, stride=1, capacity=64 ** 3)  # what any draw keeps
    box = torch.zeros(n ** 3, device="cuda")
    q = params(n, 2.19, seed=5, nbar=1e-6)
    cats = []
    for _ in range(2):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        cat, count = c.draw_qso(q, [box] * 3, stride=1, capacity=1_000_000)
        del cat
        cats.append(count)
        torch.cuda.empty_cache()
        assert free - torch.cuda.mem_get_info()[0] <= 256 << 20
    assert cats[0] == cats[1] > 10_000
    c.close()
