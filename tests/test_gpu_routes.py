"""The two fused kernels against the oracle on both sides of every rule that chooses
between them: pixel lengths around the limits of each layout and length, skewers of
one segment at most, P_s at one and at several redshifts, the tensor box among the
layouts."""
import numpy as np
import pytest

import oracle
import skewer_inputs as si
from tests.parity_util import NTHREADS, assert_field_close, assert_flux_close, assert_stats_close
from tests.test_gpu_pairs import FLAGS, check, recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2310_18996_gb300 as mk  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = mk.Context(0)
    yield c
    c.close()


def with_nodes(w, zs):
    p_s = np.stack([(0.5 + k / len(zs)) * np.asarray(w["p_s"]) for k in range(len(zs))])
    return si.shrink(w, p_s=p_s, p_s_z=list(zs))


def check_tensor(ctx, w):
    w = dict(w, eta_mode=1)
    d, e6 = si.gaussian_box_tensor(w["n"], w["cell"], w["seed_box"])
    pos, ids = si.catalogue(w)
    pos[: len(pos) // 2, 1:] *= -7.0  # steep sight lines
    o = oracle.run_skewers(w, d, e6, pos, ids, n_threads=NTHREADS)
    so = oracle.stats(w, o["j_lo"], o["offsets"], o["offsets_out"], o["flux"], o["delta"], o["eta"])
    box = ctx.load_box(w, ctx.pack_box_tensor(torch.from_numpy(d).cuda(), torch.from_numpy(e6).cuda()), None,
                       layout=mk.BOX_TENSOR)
    st, g = ctx.run(box, mk.catalogue_tensor(pos, ids), len(ids), w, flags=FLAGS)
    tot = int(o["offsets"][-1])
    np.testing.assert_array_equal(g["offsets"].cpu().numpy(), o["offsets"])
    assert_field_close(g["delta"][:tot].cpu().numpy(), o["delta"], "delta_tot")
    assert_field_close(g["eta"][:tot].cpu().numpy(), o["eta"], "eta")
    assert_flux_close(g["flux"][:tot].cpu().numpy(), o["flux"])
    one = so["sums"][:, 0] == 1  # a pixel on its own: 0, or the root of the rounding of F^2
    assert np.all((st["sigma_f"][one] >= 0) & (st["sigma_f"][one] <= 2.0 ** -11))
    st["sigma_f"][one] = so["sigma_f"][one]
    assert_stats_close(st, so)


# cells on both sides of a limit (dr = 0.2): 0.115, 0.14, 0.2, 0.25 cells a pixel, and far beyond
@pytest.mark.parametrize("n_fft,cell", [(256, 0.77), (256, 0.81), (256, 0.1), (512, 0.81), (1024, 0.79), (1024, 0.81),
                                        (2048, 0.99), (2048, 1.01)])
@pytest.mark.parametrize("nodes", [False, True])
def test_tensor(ctx, n_fft, cell, nodes):
    w = recipe(cell, n_fft=n_fft)
    check_tensor(ctx, with_nodes(w, [2.0, 2.6, 3.4]) if nodes else w)


@pytest.mark.parametrize("n_fft,cell", [(256, 1.73), (256, 1.75), (512, 1.42), (512, 1.44), (1024, 1.42), (1024, 1.44),
                                        (2048, 0.99), (2048, 1.01)])
@pytest.mark.parametrize("layout", [mk.BOX_PADDED, mk.BOX_INTERLEAVED])
def test_pixel_lengths_at_the_limits(ctx, layout, n_fft, cell):
    check(ctx, recipe(cell, n_fft=n_fft), layout)


@pytest.mark.parametrize("n_fft", [256, 512, 1024, 2048])
@pytest.mark.parametrize("layout", [mk.BOX_PLANAR, mk.BOX_INTERLEAVED, mk.BOX_PADDED, mk.BOX_HALO])
@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_skewers_of_one_segment(ctx, n_fft, layout, extra):
    w = recipe(si.CELL, n_fft=n_fft, n_max=n_fft + extra)
    check(ctx, with_nodes(w, [2.0, 2.6, 3.4]) if extra == 0 else w, layout)
