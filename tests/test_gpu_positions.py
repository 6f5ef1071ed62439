"""Where on its sight line a pixel is read: the record's own position, without a
drift along the run of pixels that shares cells."""
import numpy as np
import pytest

import skewer_inputs as si
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


def test_no_drift_at_the_end_of_a_pair():
    """delta is +1 and -1 in turn along x, so a pixel's value gives its position in
    the cell.  A pixel's weight is rounded on its own (2^-25, averaged out here); the
    slope of its cell is an FP32 number, at worst 2^-24 of the half cell that a pixel
    is from the cell's first on average: 2^-24 / (2 sqrt 3) over many skewers."""
    ctx = mk.Context(0)
    w = recipe(2.0, n_fft=2048, n_max=4096)
    w = si.shrink(w, n_q=300, lrf_min=300.0, p_s=np.zeros(1025))
    pos, ids = si.catalogue(w)
    n = len(ids)
    d = torch.ones((w["n"],) * 3)
    d[:, :, 1::2] = -1.0
    d = d.cuda()
    box = ctx.load_box(w, ctx.pack_box(d, torch.zeros_like(d), padded=True), None, layout=mk.BOX_PADDED)
    r = ctx.make_skewers(box, mk.catalogue_tensor(pos, ids), n, w)
    rec, off = mk.skewer_records(r["sk"], n), r["offsets"].cpu().numpy()
    delta = r["delta"].cpu().numpy().astype(np.float64)
    drift = []
    j = np.arange(3000, 4096)
    for q in range(n):
        assert rec["n"][q] == 4096
        x = (int(rec["p0"][q][0]) + j * int(rec["step"][q][0])) / 2.0 ** 44
        cell, t = np.floor(x), x - np.floor(x)
        sign = np.where(cell % 2 == 0, -2.0, 2.0)
        ratio = delta[off[q] + j] / (-0.5 * sign + sign * t)  # the growth factor, smooth along the line
        ok = np.abs(t - 0.5) > 0.2
        growth = np.polyval(np.polyfit(j[ok] - 3548, ratio[ok], 4), j - 3548)
        err = (delta[off[q] + j] / growth - (-0.5 * sign + sign * t)) / sign
        drift.append(np.mean(err))
    rms = np.sqrt(np.mean(np.square(drift)))
    print("rms drift %.2e cells" % rms)
    assert rms <= 2.0 ** -24 / (2 * np.sqrt(3.0))
    ctx.close()
