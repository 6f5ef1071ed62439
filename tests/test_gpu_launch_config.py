"""mk_launch_config reports a register budget that the variant's kernel has, by
default and after the autotuner has chosen."""
import numpy as np
import pytest

import skewer_inputs as si
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402

NODES, SEGMENT, GAUSS = 32, 64, 16


def test_budgets_of_the_instances():
    c = mk.Context(0)
    for n_fft in (256, 512, 1024, 2048):
        tensor = 2 if n_fft <= 1024 else 3
        for layout, budget in ((mk.BOX_TENSOR, tensor), (mk.BOX_TENSOR + NODES, tensor), (mk.BOX_PADDED, 3),
                               (mk.BOX_PADDED + NODES, 3), (mk.BOX_TENSOR + SEGMENT, 3), (mk.BOX_PLANAR + SEGMENT, 3),
                               (mk.BOX_TENSOR + SEGMENT + NODES, 3), (mk.BOX_HALO + GAUSS + NODES, 3)):
            assert c.launch_config(n_fft, layout=layout) == (256, budget, False)
    c.close()


@pytest.mark.parametrize("cell,nodes,variant", [(1.0, False, SEGMENT), (si.CELL, True, NODES)])
def test_autotuner_records_an_instance(cell, nodes, variant):
    c = mk.Context(0)
    w = recipe(cell, n_fft=256)
    if nodes:
        w = si.shrink(w, p_s=np.stack([w["p_s"]] * 2), p_s_z=[2.0, 3.0])
    pos, ids = si.catalogue(w)
    d = torch.randn((w["n"],) * 3, device="cuda")
    box = c.load_box(w, c.pack_box(d, d, padded=True), None, layout=mk.BOX_PADDED)
    c.run(box, mk.catalogue_tensor(pos, ids), len(ids), w, flags=mk.STATS | mk.AUTOTUNE)
    threads, budget, tuned = c.launch_config(256, layout=mk.BOX_PADDED + variant)
    assert tuned and budget == 3 and threads in (128, 256)
    c.close()
