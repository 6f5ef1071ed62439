"""A captured step is replayed only for the kernel it was captured with: the two
interpolations of one halo box, in turn into the same buffers."""
import numpy as np
import pytest

import skewer_inputs as si
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


@pytest.mark.parametrize("cell", [1.0, si.CELL])  # gathers per pixel, and cells
def test_interpolations_in_turn(cell):
    c = mk.Context(0)
    w = recipe(cell, n_fft=256)
    g = si.shrink(w, interp=mk.INTERP_GAUSS7)
    pos, ids = si.catalogue(w)
    n, q = len(ids), mk.catalogue_tensor(pos, ids)
    d = torch.randn((w["n"],) * 3, device="cuda")
    box = c.load_box(w, c.pack_box(d, d, halo=True), None, layout=mk.BOX_HALO)
    flags = mk.STATS | mk.STORE_FLUX
    want = [c.run(box, q, n, x, flags=flags)[1]["flux"].clone() for x in (w, g)]
    assert not torch.equal(*want)
    _, _, total = c.plan(box, q, n, w)
    out = None
    with torch.cuda.stream(torch.cuda.Stream()):
        for x, f in zip((w, g, w, g), want * 2):
            _, out = c.run(box, q, n, x, flags=flags | mk.GRAPH, capacity=total, outputs=out)
            torch.cuda.synchronize()
            assert torch.equal(out["flux"][:total], f[:total])
    c.close()
