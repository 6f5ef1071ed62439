"""A value that is not finite, or far larger than the rest, spoils the statistics
of its own segment and pixel and of nothing else: segments that share a
transform do not share their values."""
import numpy as np
import pytest

import oracle
import skewer_inputs as si
from tests.parity_util import NTHREADS, TOL_STAT, box_numpy
from tests.test_gpu_pairs import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = mk.Context(0)
    yield c
    c.close()


def stored(ctx, n_fft, rebin):
    """Skewers of three segments and a bit, narrow z bins (a segment has about one of its own)."""
    w = recipe(si.CELL, n_fft=n_fft, n_max=rebin * (3 * n_fft + n_fft // 3))
    w = si.shrink(w, n_q=24, lrf_min=300.0, n_zbins=32, z_bin_lo=0.4, dz_bin=0.1)
    d, e = box_numpy(w)
    pos, ids = si.catalogue(w)
    o = oracle.run_skewers(w, d, e, pos, ids, rebin=rebin, n_threads=NTHREADS)
    box = ctx.load_box(w, torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda())
    r = ctx.make_skewers(box, mk.catalogue_tensor(pos, ids), len(ids), w)
    f, off = ctx.flux(w, r["sk"], len(ids), r["delta"], r["eta"], rebin=rebin)
    return w, o, r, f, off


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e12, -1e7, 1e-12])
@pytest.mark.parametrize("n_fft,rebin", [(256, 1), (256, 3), (512, 1), (1024, 1), (2048, 1)])
def test_stored_flux(ctx, n_fft, rebin, value):
    w, o, r, f, off = stored(ctx, n_fft, rebin)
    f, n = f.cpu().numpy()[: o["offsets_out"][-1]], len(o["j_lo"])
    for q in range(n):  # in the first, second, third and trailing segment; 1e-12: a whole segment
        a, b = o["offsets_out"][q] + (q % 4) * n_fft, o["offsets_out"][q + 1]
        if q % 6 < 4 and a < b:
            f[a + min(q, b - a - 1)] = value
            if value == 1e-12:
                f[a: min(a + n_fft, b)] *= np.float32(value)
    ref = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], f.astype(np.float64), o["delta"], o["eta"],
                       rebin=rebin)
    got = ctx.stats(w, r["sk"], n, off, torch.from_numpy(f).cuda(), rebin=rebin, delta=r["delta"], eta=r["eta"])
    np.testing.assert_array_equal(got["n_seg"], ref["n_seg"])
    p, g = ref["p1d_sum"], got["p1d_sum"]
    assert np.isfinite(p).any() and (np.isfinite(value) or not np.isfinite(p).all())
    np.testing.assert_array_equal(np.isfinite(g), np.isfinite(p))
    m = np.isfinite(p)
    np.testing.assert_allclose(g[m], p[m], rtol=TOL_STAT)


@pytest.mark.parametrize("n_fft", [256, 512, 1024, 2048])
def test_tuning_pass_and_fused(ctx, n_fft):
    """NaN pixels of stored fields (staged or not), and a NaN voxel of the box."""
    w, o, r, _, _ = stored(ctx, n_fft, 1)
    n, delta = len(o["j_lo"]), r["delta"].clone()
    flux = o["flux"].copy()
    for q in range(0, n, 4):
        a, b = o["offsets"][q] + (q // 4 % 4) * n_fft, o["offsets"][q + 1]
        if a < b:
            delta[a] = float("nan")
            flux[a] = np.nan
    ref = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], flux, o["delta"], o["eta"])["p1d_sum"]
    odd = [torch.cat([torch.zeros(1, device="cuda"), x])[1:] for x in (delta, r["eta"])]
    for x in ((delta, r["eta"]), odd):
        got = ctx.flux_stats(w, r["sk"], n, r["offsets"], *x)["p1d_sum"]
        m = np.isfinite(ref)
        assert m.any() and not m.all()
        np.testing.assert_array_equal(np.isfinite(got), m)
        np.testing.assert_allclose(got[m], ref[m], rtol=TOL_STAT)
    d, e = box_numpy(w)
    d[:, :, 5] = np.nan  # a plane across the sight lines
    pos, ids = si.catalogue(w)
    o = oracle.run_skewers(w, d, e, pos, ids, n_threads=NTHREADS)
    ref = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], o["flux"], o["delta"], o["eta"])["p1d_sum"]
    box = ctx.load_box(w, ctx.pack_box(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda(), padded=True), None,
                       layout=mk.BOX_PADDED)
    got = ctx.run(box, mk.catalogue_tensor(pos, ids), n, w)[0]["p1d_sum"]
    m = np.isfinite(ref)
    np.testing.assert_array_equal(np.isfinite(got), m)
    np.testing.assert_allclose(got[m], ref[m], rtol=TOL_STAT)
