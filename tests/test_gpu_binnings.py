"""Statistics at the ends of the binnings: one k bin (fewer than a team has warps)
to 64, one z bin to 32, the CTAs that the accumulators leave room for, in the fused
pass, the tuning pass and the statistics of stored flux."""
import numpy as np
import pytest

import oracle
import skewer_inputs as si
from tests.parity_util import NTHREADS, assert_stats_close, box_numpy
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


def faint_bins(s, so, key):
    """An FP32 transform rounds at ~5e-7 of its largest amplitude, so a k bin of a mode or two
    below 1e-4 of the largest power P_m is known to 1e-6 sqrt(P P_m), not to 1e-4 P (one set of
    transforms per segment fails there at four of these sizes, the pair transform at one)."""
    p, m = so[key], so[key].max(axis=1, keepdims=True)
    faint = p < 1e-4 * m
    assert np.all(np.abs(s[key] - p)[faint] <= 1e-6 * np.sqrt(p * m)[faint])
    return np.where(faint, p, s[key])


@pytest.mark.parametrize("n_fft,n_z,n_k", [(256, 1, 1), (256, 12, 64), (256, 20, 32), (256, 32, 32), (256, 32, 64),
                                           (512, 16, 64), (512, 32, 64), (512, 3, 1), (1024, 16, 32), (1024, 32, 64),
                                           (1024, 5, 2), (1024, 2, 1), (2048, 32, 64), (2048, 7, 4), (2048, 3, 1),
                                           (2048, 4, 8)])
def test_binnings(n_fft, n_z, n_k):
    ctx = mk.Context(0)
    w = recipe(si.CELL, n_fft=n_fft, n_max=2 * n_fft + 300)
    w = si.shrink(w, n_q=40, lrf_min=500.0, n_zbins=n_z, z_bin_lo=1.5, dz_bin=2.4 / n_z, n_kbins=n_k)
    d, e = box_numpy(w)
    pos, ids = si.catalogue(w)
    n = len(ids)
    box = ctx.load_box(w, torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda())
    cat = mk.catalogue_tensor(pos, ids)
    for rebin in (1, 2):
        o = oracle.run_skewers(w, d, e, pos, ids, rebin=rebin, n_threads=NTHREADS)
        so = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], o["flux"], o["delta"], o["eta"], rebin=rebin)
        r = ctx.make_skewers(box, cat, n, w)
        f, off = ctx.flux(w, r["sk"], n, r["delta"], r["eta"], rebin=rebin)
        st = ctx.stats(w, r["sk"], n, off, f, rebin=rebin, delta=r["delta"], eta=r["eta"])
        one = so["sums"][:, 0] == 1  # (a pixel on its own has no dispersion)
        for s in ([st] if rebin > 1 else [st, ctx.run(box, cat, n, w)[0]]):
            assert np.all((s["sigma_f"][one] >= 0) & (s["sigma_f"][one] <= 2.0 ** -11))
            s["sigma_f"][one] = so["sigma_f"][one]
            s["p1d_f"], s["p1d_df"] = faint_bins(s, so, "p1d_f"), faint_bins(s, so, "p1d_df")
            assert_stats_close(s, so)
        if rebin == 1:
            tp = ctx.flux_stats(w, r["sk"], n, r["offsets"], r["delta"], r["eta"])
            for k in ("sums", "p1d_sum", "n_seg"):
                np.testing.assert_array_equal(tp[k], st[k])
    ctx.close()
