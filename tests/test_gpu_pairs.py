"""The fused kernel's pairs of segments and cells of a sight line against the
oracle: skewer lengths around the ends of segments and pairs, pixel lengths on
both sides of the rule that chooses cells or gathers per pixel, every layout."""
import numpy as np
import pytest

import oracle
import skewer_inputs as si
from tests.parity_util import NTHREADS, assert_field_close, assert_flux_close, assert_stats_close, box_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402

FLAGS = mk.STATS | mk.STORE_FIELDS | mk.STORE_FLUX


@pytest.fixture(scope="module")
def ctx():
    c = mk.Context(0)
    yield c
    c.close()


def recipe(cell, **kw):
    w = si.shrink(si.workload("tiny"), n_q=60, **kw)
    half = 0.5 * w["n"] * cell
    w.update(cell=cell, origin=(si.OBSERVER_TO_BOX_CENTRE - half, -half, -half))
    return w


def check(ctx, w, layout):
    d, e = box_numpy(w)
    pos, ids = si.catalogue(w)
    pos[: len(pos) // 2, 1:] *= -7.0  # steep sight lines, both directions along y and z
    o = oracle.run_skewers(w, d, e, pos, ids, n_threads=NTHREADS)
    so = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], o["flux"], o["delta"], o["eta"])
    gd, ge = torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda()
    if layout == mk.BOX_PLANAR:
        box = ctx.load_box(w, gd, ge)
    else:
        packed = ctx.pack_box(gd, ge, padded=layout == mk.BOX_PADDED, halo=layout == mk.BOX_HALO)
        box = ctx.load_box(w, packed, None, layout=layout)
    st, g = ctx.run(box, mk.catalogue_tensor(pos, ids), len(ids), w, flags=FLAGS)
    tot = int(o["offsets"][-1])
    np.testing.assert_array_equal(g["offsets"].cpu().numpy(), o["offsets"])
    assert_field_close(g["delta"][:tot].cpu().numpy(), o["delta"], "delta_tot")
    assert_field_close(g["eta"][:tot].cpu().numpy(), o["eta"], "eta")
    assert_flux_close(g["flux"][:tot].cpu().numpy(), o["flux"])
    one = so["sums"][:, 0] == 1  # one pixel has no dispersion: 0, or the root of a rounding error
    st["sigma_f"][one] = so["sigma_f"][one]
    assert_stats_close(st, so)


@pytest.mark.parametrize("n_fft,n_max", [(256, n) for n in (1, 31, 255, 256, 257, 511, 512, 513, 769)] +
                         [(512, 513), (1024, 1025), (2048, 1900)])
def test_segment_and_pair_ends(ctx, n_fft, n_max):
    check(ctx, recipe(si.CELL, n_fft=n_fft, n_max=n_max), mk.BOX_PADDED)


@pytest.mark.parametrize("cell", [0.3, 1.0, 1.99, 2.0, 9.0])  # dr/cell 0.67 ... 0.1005, 0.1, 0.022
@pytest.mark.parametrize("n_fft", [256, 2048])
def test_pixel_lengths_on_both_sides_of_the_cell_rule(ctx, cell, n_fft):
    check(ctx, recipe(cell, n_fft=n_fft), mk.BOX_PADDED)


@pytest.mark.parametrize("layout", [mk.BOX_PLANAR, mk.BOX_INTERLEAVED, mk.BOX_HALO])
@pytest.mark.parametrize("cell", [1.5, 2.0])
def test_layouts_with_and_without_cells(ctx, layout, cell):
    check(ctx, recipe(cell, n_fft=512, n_max=1500), layout)


@pytest.mark.parametrize("n_fft,n_max,rebin", [(256, n, 1) for n in (255, 256, 257, 512, 513, 769)] +
                         [(512, 1025, 1), (2048, 1900, 1), (256, 514, 2), (256, 1500, 5), (512, 1537, 3)])
def test_statistics_at_pair_ends(ctx, n_fft, n_max, rebin):
    """Statistics of stored flux at any rebin, and the tuning pass with its
    fields staged and not, at lengths around the ends of segments and pairs."""
    w = recipe(si.CELL, n_fft=n_fft, n_max=n_max)
    d, e = box_numpy(w)
    pos, ids = si.catalogue(w)
    n = len(ids)
    o = oracle.run_skewers(w, d, e, pos, ids, rebin=rebin, n_threads=NTHREADS)
    so = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], o["flux"], o["delta"], o["eta"], rebin=rebin)
    box = ctx.load_box(w, torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda())
    r = ctx.make_skewers(box, mk.catalogue_tensor(pos, ids), n, w)
    f, off = ctx.flux(w, r["sk"], n, r["delta"], r["eta"], rebin=rebin)
    st = ctx.stats(w, r["sk"], n, off, f, rebin=rebin, delta=r["delta"], eta=r["eta"])
    assert_stats_close(st, so)
    if rebin == 1:
        odd = [torch.cat([torch.zeros(1, device="cuda"), x])[1:] for x in (r["delta"], r["eta"])]
        for x in ((r["delta"], r["eta"]), odd):
            tp = ctx.flux_stats(w, r["sk"], n, r["offsets"], *x)
            for k in ("sums", "p1d_sum", "n_seg"):
                np.testing.assert_array_equal(tp[k], st[k])


@pytest.mark.parametrize("n_fft,n_max,cell", [(256, n, 9.0) for n in (1, 3, 5, 255, 257, 769)] +
                         [(256, 1500, c) for c in (0.3, 2.0)] + [(1024, 742, 2.0), (2048, 1900, 0.3), (2048, 7, 2.0)])
def test_gaussian_kernel_runs(ctx, n_fft, n_max, cell):
    """Runs of pixels in one voxel: of one pixel (a voxel a pixel) to many, cut
    by the ends of segments, with fewer runs than warps and more than lanes."""
    check(ctx, recipe(cell, n_fft=n_fft, n_max=n_max, interp=mk.INTERP_GAUSS7), mk.BOX_HALO)


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 6145, 4096 * 2048, 4096 * 2048 + 2049])
def test_offsets_at_the_tiles_of_the_scan(ctx, n):
    """Offsets are the running sum of the lengths, for one tile, a few, and past
    the number of tiles whose sums are scanned in a launch of their own."""
    w = recipe(si.CELL, n_fft=256, n_max=0)
    pos, ids = si.catalogue(si.shrink(w, n_q=min(n, 4099)))
    k = -(-n // len(ids))
    q = mk.catalogue_tensor(pos, ids).repeat(k)[: n * mk.QSO_DTYPE.itemsize]
    z = torch.zeros((w["n"],) * 3, device="cuda")
    sk, offsets, total = ctx.plan(ctx.load_box(w, z, z), q, n, w)
    lengths = torch.from_numpy(mk.skewer_records(sk, n)["n"].astype(np.int64))
    assert int(lengths.sum()) == total
    np.testing.assert_array_equal(offsets.cpu().numpy(), np.concatenate([[0], np.cumsum(lengths.numpy())]))


@pytest.mark.parametrize("zs", [[2.2, 2.9], list(np.linspace(1.9, 3.6, 32)), [0.5, 1.0, 1.5], [5.0, 6.0, 7.0]])
@pytest.mark.parametrize("n_max", [0, 300])
def test_p_s_nodes_around_the_segments(ctx, zs, n_max):
    """The fewest and the most nodes, and segments below and above all of them."""
    w = recipe(si.CELL, n_max=n_max)
    p_s = np.stack([(0.5 + k / len(zs)) * np.asarray(w["p_s"]) for k in range(len(zs))])
    check(ctx, si.shrink(w, p_s=p_s, p_s_z=zs), mk.BOX_PADDED)
