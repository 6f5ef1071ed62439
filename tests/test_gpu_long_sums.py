"""Sums of many pixels into one z bin by few CTAs, against 64-bit sums of the same
pixels.  A thread adds its pixels in FP32 over a bounded run, and runs are added
with compensation, so the errors of the runs are independent and average out: what
is left is the rounding of a compensated sum, a few units of 2^-24."""
import numpy as np
import pytest

import skewer_inputs as si
from tests.parity_util import box_numpy
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402

TOL = 4 * 2.0 ** -24


def check(sums, f, d, e):
    s = sums[0]
    n = f.numel()
    assert s[0] == n
    f, d, e = f.double(), d.double(), e.double()
    want = [f.sum(), (f * f).sum(), d.sum(), e.sum(), (d * d).sum(), (e * e).sum(), (d * e).sum(), (f * d).sum(),
            (f * e).sum()]
    rms = [x.norm().item() for x in (f, d, e)]
    root = n ** 0.5
    size = [rms[0] * root, rms[0] ** 2, rms[1] * root, rms[2] * root, rms[1] ** 2, rms[2] ** 2, rms[1] * rms[2],
            rms[0] * rms[1], rms[0] * rms[2]]
    err = [abs(a - b.item()) / c for a, b, c in zip(s[1:10], want, size)]
    print(["%.1e" % x for x in err])
    assert max(err) <= TOL, err


@pytest.mark.parametrize("n_fft", [256, 1024])
def test_one_wide_bin(n_fft):
    ctx = mk.Context(0)
    w = recipe(si.CELL, n_fft=n_fft, n_max=1500)
    w = si.shrink(w, n_q=40000, n_zbins=1, z_bin_lo=0.0, dz_bin=12.0)
    w["seed_cat"] = 77
    pos, ids = si.catalogue(w)
    q, n = mk.catalogue_tensor(pos, ids), len(ids)
    d, e = (torch.from_numpy(x).cuda() for x in box_numpy(w))
    box = ctx.load_box(w, ctx.pack_box(d, e, padded=True), None, layout=mk.BOX_PADDED)
    ctx.set_grid_cap(1)
    st, o = ctx.run(box, q, n, w, flags=mk.STATS | mk.STORE_FLUX | mk.STORE_FIELDS)
    tot = int(o["offsets"][-1])
    delta, eta, flux = (o[k][:tot] for k in ("delta", "eta", "flux"))
    check(st["sums"], flux, delta, eta)
    st = ctx.flux_stats(w, o["sk"], n, o["offsets"], delta, eta)
    check(st["sums"], flux, delta, eta)
    for rebin in (1, 3):
        f, off = ctx.flux(w, o["sk"], n, delta, eta, rebin=rebin)
        st = ctx.stats(w, o["sk"], n, off, f, rebin=rebin, delta=delta, eta=eta)
        # the fine pixels of every output pixel
        m = (o["offsets"][1:] - o["offsets"][:-1]) // rebin
        first = torch.repeat_interleave(o["offsets"][:-1] - rebin * off[:-1], m)
        at = first + rebin * torch.arange(int(off[-1]), device="cuda")
        mean = [sum(x[at + r].double() for r in range(rebin)) / rebin for x in (delta, eta)]
        check(st["sums"], f[: int(off[-1])], *mean)
    ctx.close()
