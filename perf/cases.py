"""Performance cases: what users of this library have it do, through its public entry points.

Each case is one call (or the two calls that belong together) of the Python binding, on
inputs made on the GPU from a seed: a Gaussian box with the power spectrum the benchmark
uses, a quasar catalogue over its redshift range, the paper's pixel length and statistic
bins.  `exact` computes the same outputs in 64 bits with torch and numpy alone.
"""
import math

import numpy as np
import torch

import paper_2310_18996_gb300 as mk

OMEGA_M, LAMBDA_LYA, C_H0 = 0.3147, 1215.67, 2997.92458
CELL, DR, CENTRE = 2.19, 0.2, 3800.0       # h^-1 Mpc: voxel, pixel, observer to box centre
NODE_Z = [1.8 + 0.2 * i for i in range(12)]  # FGPA nodes and z-bin centres
X_RANGE = (3620.44, 4943.61)               # quasar distances, z 2.04 - 4.0
THIN = 10_000                              # bins with fewer pixels carry no sigma_F, b_F, beta_F


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a quick look while setting up a mock: 64^3 box, 500 sight lines, flux and statistics
        {"name": "fused tiny", "kind": "fused", "n": 64, "n_q": 500, "n_fft": 256, "layout": "padded",
         "n_max": 0, "ps_nodes": 1, "store": True, "graph": False},
        # the production pass: 1024^3 box, 1M quasars, skewers of 200 - 1500 pixels
        {"name": "fused survey", "kind": "fused", "n": 1024, "n_q": 1_000_000, "n_fft": 256, "layout": "padded",
         "n_max": 1500, "ps_nodes": 1, "store": True, "graph": True},
        # one pass of the paper's P_S tuning: statistics only, P_S given at the z nodes
        {"name": "P_S tuning pass", "kind": "fused", "n": 512, "n_q": 100_000, "n_fft": 1024, "layout": "padded",
         "n_max": 0, "ps_nodes": 12, "store": False, "graph": False},
        # the velocity gradient along the true sight line, from six boxes
        {"name": "radial eta", "kind": "fused", "n": 512, "n_q": 100_000, "n_fft": 256, "layout": "tensor",
         "n_max": 1500, "ps_nodes": 1, "store": True, "graph": False},
        # the paper's own interpolation, a Gaussian kernel over 7^3 voxels
        {"name": "Gaussian kernel", "kind": "fused", "n": 512, "n_q": 100_000, "n_fft": 256, "layout": "gauss7",
         "n_max": 1500, "ps_nodes": 1, "store": True, "graph": False},
        # saved pre-production: delta and eta of full forests, one delta_S realisation per ~skewer
        {"name": "pre-production", "kind": "make", "n": 512, "n_q": 100_000, "n_fft": 2048, "layout": "padded",
         "n_max": 0},
        # the pass that tuning a, b, c repeats: FGPA of stored skewers and their statistics
        {"name": "tuning pass", "kind": "tune", "n_q": 1_000_000, "n_fft": 256, "n_max": 1500},
        # post-production at spectrograph pixels: FGPA and rebin by 3, then the statistics
        {"name": "rebinned spectra", "kind": "rebin", "n_q": 100_000, "n_fft": 256, "n_max": 1500, "rebin": 3},
        # catalogue from and flux to page-locked host memory, pipelined
        {"name": "host pipeline", "kind": "host", "n": 512, "n_q": 100_000, "n_fft": 256, "n_max": 1500,
         "chunks": 8},
        # a new realisation of the boxes
        {"name": "box synthesis", "kind": "synth", "n": 1024, "cell": CELL, "layout": "padded"},
        # quasars from three lognormal quasar-density boxes
        {"name": "quasar draw", "kind": "draw", "n": 512, "cell": CELL, "nbar": 1e-4},
        # some training steps of the tuning surrogate
        {"name": "surrogate training", "kind": "train", "n_samples": 5632, "batch": 256, "epochs": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fused", "fused", "fused", "make", "tune", "rebin", "host", "synth", "draw", "train"])
    c = {"kind": kind}
    if kind in ("fused", "make", "host"):
        layout = rng.choice(["padded", "padded", "tensor", "gauss7"]) if kind == "fused" else "padded"
        c.update(n=rng.choice([64, 128, 256, 512]), n_q=_log(rng, 200, 60_000 if layout == "gauss7" else 200_000),
                 n_fft=rng.choice([256, 256, 512, 1024, 2048]), n_max=rng.choice([0, rng.randint(300, 1500)]))
    if kind == "fused":
        c.update(layout=layout, ps_nodes=rng.choice([1, 1, 1, rng.randint(2, 12)]), store=rng.random() < 0.7,
                 graph=rng.random() < 0.3)
    elif kind == "make":
        c.update(layout="padded")
    elif kind == "tune":
        c.update(n_q=_log(rng, 500, 1_000_000), n_fft=rng.choice([256, 256, 512, 1024]),
                 n_max=rng.randint(300, 1500))
    elif kind == "rebin":
        c.update(n_q=_log(rng, 500, 300_000), n_fft=256, n_max=rng.randint(300, 1500), rebin=rng.randint(1, 5))
    elif kind == "host":
        c.update(chunks=rng.choice([4, 8, 16]))
    elif kind == "synth":
        c.update(n=rng.choice([128, 256, 512, 512, 1024]), cell=round(rng.uniform(1.5, 3.0), 3),
                 layout=rng.choice(["padded", "padded", "planar", "halo", "tensor"]))
        if c["n"] == 1024 and c["layout"] == "tensor":
            c["n"] = 512
    elif kind == "draw":
        c.update(n=rng.choice([128, 256, 512]), cell=round(rng.uniform(1.5, 3.0), 3),
                 nbar=math.exp(rng.uniform(math.log(2e-5), math.log(1e-3))))
    elif kind == "train":
        c.update(n_samples=_log(rng, 300, 20_000), batch=256, epochs=1)
    return c


# ------------------------------------------------------------------ recipes and inputs
def _recipe(case, seed):
    n, n_fft = case.get("n", 512), case.get("n_fft", 256)
    side = n * CELL
    m = np.arange(n_fft // 2 + 1)
    k = 2.0 * np.pi * m / (n_fft * DR)
    with np.errstate(divide="ignore"):
        p_s = 0.1 / k * np.exp(-(k / 5.0) ** 2)
    p_s[0] = 0.0
    w = dict(n=n, cell=CELL, origin=(CENTRE - 0.5 * side, -0.5 * side, -0.5 * side), dr=DR, lrf_min=1040.0,
             lrf_max=1200.0, lobs_min=3600.0 if case.get("n_max") else 0.0, n_min=200 if case.get("n_max") else 0,
             n_max=case.get("n_max", 0), n_fft=n_fft, seed_noise=(3003 + seed) & 0xFFFFFFFF, node_z=list(NODE_Z),
             node_ln_a=[math.log(0.01) + 4.0 * math.log(1.0 + z) for z in NODE_Z], node_b=[1.6] * 12,
             node_c=[1.0] * 12, n_zbins=12, z_bin_lo=1.7, dz_bin=0.2, n_kbins=32, n_fft_p1d=n_fft)
    nodes = case.get("ps_nodes", 1)
    if nodes > 1:  # amplitude falling with z, as tuned tables do
        w["p_s_z"] = np.linspace(1.8, 4.0, nodes)
        p_s = np.concatenate([p_s * (1.4 - 0.2 * z) for z in w["p_s_z"]])
    w["p_s"] = p_s
    if case.get("layout") == "gauss7":
        w["interp"] = mk.INTERP_GAUSS7
    return w


def _rng(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 7919 + what) & 0x7FFFFFFF)
    return g


def _spectrum(k):
    """3D power spectrum of the boxes (unnormalised)."""
    return torch.where(k > 0, k.clamp_min(1e-9) ** 0.96 * torch.exp(-(k / 1.5) ** 2)
                       * (1.0 + 0.05 * torch.sin(150.0 * k)), torch.zeros_like(k))


def _box(n, seed, pairs):
    """Gaussian box of unit variance and, per (a, b) of pairs, IFFT[-(k_a k_b / k^2) delta_k]."""
    f = torch.fft.rfftn(torch.randn((n, n, n), generator=_rng(seed, 1), device="cuda"))
    kx = 2.0 * math.pi * torch.fft.rfftfreq(n, d=CELL, device="cuda")
    ky = 2.0 * math.pi * torch.fft.fftfreq(n, d=CELL, device="cuda")
    ks = (kx[None, None, :], ky[None, :, None], ky[:, None, None])
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    p = _spectrum(torch.sqrt(k2))
    both = torch.full((n // 2 + 1,), 2.0, device="cuda")
    both[0] = both[-1] = 1.0
    f *= torch.sqrt(p * (n ** 3 / (p * both).sum(dtype=torch.float64)).float())
    del p
    delta = torch.fft.irfftn(f, s=(n, n, n))
    f /= -torch.where(k2 > 0, k2, torch.ones_like(k2))
    return delta, [torch.fft.irfftn(f * (ks[a] * ks[b]), s=(n, n, n)) for a, b in pairs]


XX = [(0, 0)]
SIX = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


def _catalogue(case, seed):
    """Positions (FP64) and ids: uniform across the box face, at distances that cover the redshift
    range evenly in an order of their own (every seed's skewers have the same lengths, so that
    buffers keep their sizes)."""
    n_q, side = case["n_q"], case.get("n", 512) * CELL
    at = torch.randperm(n_q, generator=_rng(0, 5), device="cuda").double()
    r = X_RANGE[0] + (at + 0.5) / n_q * (X_RANGE[1] - X_RANGE[0])
    u = torch.rand((n_q, 3), generator=_rng(seed, 2), device="cuda", dtype=torch.float64)
    pos = (u - 0.5) * side
    pos[:, 0] = r
    pos *= (r / pos.norm(dim=1))[:, None]
    return pos, torch.arange(n_q, device="cuda") + 1000 * (seed % 1000)


def _records(pos, ids):
    """mk_qso records as bytes."""
    return torch.cat([pos.view(torch.int64), ids[:, None]], 1).contiguous().view(torch.uint8).reshape(-1)


def _stored_fields(total, seed):
    """delta_tot and eta of stored skewers: large-scale cells of 11 pixels plus small-scale noise."""
    g = _rng(seed, 3)
    a = torch.randn(total // 11 + 1, generator=g, device="cuda")
    b = torch.randn(total // 11 + 1, generator=g, device="cuda")
    d = torch.randn(total, generator=g, device="cuda").mul_(0.33)
    d += (0.37 * a)[:, None].expand(-1, 11).reshape(-1)[:total]
    return d, (-0.17 * a + 0.13 * b)[:, None].expand(-1, 11).reshape(-1)[:total].contiguous()


def _pk_table(cell):
    """P(k) table of the box synthesis: unit variance at about the benchmark's voxel."""
    dk, m = 0.002, 4096
    k = np.arange(m) * dk
    with np.errstate(divide="ignore", invalid="ignore"):
        p = np.where(k > 0, k ** 0.96 * np.exp(-(k / 1.5) ** 2) * (1.0 + 0.05 * np.sin(150.0 * k)), 0.0)
    return p * 2.0 * math.pi ** 2 / (np.sum(p * k * k) * dk), dk


LAYOUTS = {"padded": mk.BOX_PADDED, "tensor": mk.BOX_TENSOR, "gauss7": mk.BOX_HALO, "halo": mk.BOX_HALO,
           "planar": mk.BOX_PLANAR}


def _load_box(ctx, case, w, seed):
    delta, eta = _box(case["n"], seed, SIX if case.get("layout") == "tensor" else XX)
    layout = LAYOUTS[case.get("layout", "padded")]
    if layout == mk.BOX_TENSOR:
        packed = ctx.pack_box_tensor(delta, torch.stack(eta))
    else:
        packed = ctx.pack_box(delta, eta[0], padded=layout == mk.BOX_PADDED, halo=layout == mk.BOX_HALO)
    return ctx.load_box(w, packed, None, layout=layout)


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind, "stream": torch.cuda.Stream()}
    ctx = st["ctx"] = mk.Context()
    if kind == "synth":
        st["pk"], st["dk"] = _pk_table(case["cell"])
        st["seed"] = seed
        st["work"] = torch.empty(2 * case["n"] ** 3, device="cuda")
    elif kind == "draw":
        n = case["n"]
        f, _ = _box(n, seed, [])
        st["boxes"] = [(f * s).reshape(-1) for s in (0.9, 1.0, 1.1)]
        half = 0.5 * n * case["cell"]
        st["q"] = dict(n=n, cell=case["cell"], origin=(CENTRE + 400.0 - half, -half, -half), z_box=(1.9, 2.75, 3.6),
                       bias=(3.7, 2.33, 1.7), xi_m5=0.6, nbar=[case["nbar"]] * 40, nbar_z0=0.5, nbar_dz=0.25,
                       seed=seed)
        st["room"] = int(1.5 * case["nbar"] * (n * case["cell"]) ** 3) + 4096
    elif kind == "train":
        g = _rng(seed, 4)
        x = torch.randn((case["n_samples"], 4), generator=g, device="cuda")
        a, b = torch.randn((4, 35), generator=g, device="cuda"), torch.randn((4, 35), generator=g, device="cuda")
        st["x"], st["t"] = x, torch.tanh(x @ a) + 0.3 * torch.sin(x @ b)
        st["mlp"] = mk.Mlp(ctx, max_batch=case["batch"], seed=seed)
        st["p0"] = st["mlp"].get_params()[0]
        st["seed"] = seed
    else:
        w = st["w"] = _recipe(case, seed)
        pos, ids = _catalogue(case, seed)
        n_q = st["n_q"] = case["n_q"]
        qso = st["qso"] = _records(pos, ids)
        if kind in ("tune", "rebin"):
            box = ctx.load_box(w, torch.zeros(2, device="cuda"), None)  # geometry alone
        else:
            box = st["box"] = _load_box(ctx, case, w, seed)
        sk, off, total = ctx.plan(box, qso, n_q, w)
        st["total"] = total
        out = st["out"] = {"sk": sk, "offsets": off}
        if kind in ("tune", "rebin"):
            st["delta"], st["eta"] = _stored_fields(total, seed)
            # skewers drop their incomplete rebinned pixels: the buffer's end stays unused
            st["total_out"] = int(((off[1:] - off[:-1]) // case.get("rebin", 1)).sum())
        elif kind == "host":
            st["qso"] = qso.cpu().pin_memory()
            st["flux"] = torch.empty(total, pin_memory=True)
        elif case.get("store"):
            out["flux"] = torch.empty(max(total, 1), device="cuda")
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ run
def _statistics(s):
    """Counts as integers; the sums and what follows from them in FP32, the precision of the terms
    they add (pixels and powers are FP32, as are the accumulators)."""
    thick = s["sums"][:, 0] >= THIN
    r = {"pixels": s["sums"][:, 0].astype(np.int64), "segments": s["n_seg"].astype(np.int64),
         "sums": s["sums"][:, 1:].astype(np.float32), "p1d": s["p1d_df"].astype(np.float32),
         "mean_flux": s["mean_flux"].astype(np.float32)}
    for k in ("sigma_f", "b_f", "beta_f"):
        r[k] = np.where(thick, s[k], 0.0).astype(np.float32)
    return r


def run(st):
    kind, ctx, case = st["kind"], st["ctx"], st["case"]
    if kind == "fused":
        flags = mk.STATS | (mk.STORE_FLUX if case["store"] else 0) | (mk.AUTOTUNE | mk.GRAPH if case["graph"] else 0)
        with torch.cuda.stream(st["stream"]):
            s, o = ctx.run(st["box"], st["qso"], st["n_q"], st["w"], flags=flags, capacity=max(st["total"], 1),
                           outputs=st["out"])
        r = _statistics(s)
        r["offsets"] = o["offsets"]
        if case["store"]:
            r["flux"] = o["flux"][: st["total"]]
        return r
    if kind == "make":
        r = ctx.make_skewers(st["box"], st["qso"], st["n_q"], st["w"])
        return {"sk": r["sk"], "offsets": r["offsets"], "delta": r["delta"], "eta": r["eta"]}
    if kind == "tune":
        return _statistics(ctx.flux_stats(st["w"], st["out"]["sk"], st["n_q"], st["out"]["offsets"], st["delta"],
                                          st["eta"]))
    if kind == "rebin":
        f, off = ctx.flux(st["w"], st["out"]["sk"], st["n_q"], st["delta"], st["eta"], rebin=case["rebin"])
        r = _statistics(ctx.stats(st["w"], st["out"]["sk"], st["n_q"], off, f, rebin=case["rebin"],
                                  delta=st["delta"], eta=st["eta"]))
        r["offsets"] = off
        r["flux"] = f[: st["total_out"]]
        return r
    if kind == "host":
        s, total = ctx.run_host(st["box"], st["qso"], st["n_q"], st["w"], st["flux"], n_chunks=case["chunks"])
        r = _statistics(s)
        r["flux"] = st["flux"][:total]
        return r
    if kind == "synth":
        return ctx.synth_box(case["n"], case["cell"], st["seed"], st["pk"], st["dk"],
                             layout=LAYOUTS[case["layout"]], work=st["work"])
    if kind == "draw":
        cat, count = ctx.draw_qso(st["q"], st["boxes"], stride=1, capacity=st["room"])
        room = torch.zeros(st["room"] * mk.QSO_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        room[: len(cat)] = cat  # into the program's catalogue array, of one size for all realisations
        return {"catalogue": room, "count": count}
    mlp = st["mlp"]
    mlp.set_params(st["p0"])
    loss = mlp.train(st["x"], st["t"], batch=case["batch"], epochs=case["epochs"], lr=2e-3, seed=st["seed"])
    return {"weights": mlp.get_params()[0], "loss": loss.astype(np.float32)}


# ------------------------------------------------------------------ work
def _mean_pixels(case):
    """Pixels per sight line, about: the forest is 1760 - 2240 pixels, cut at n_max."""
    return min(1900, case["n_max"] or 1900) * (0.96 if case["n_max"] else 1.0)


def work(case):
    kind = case["kind"]
    if kind in ("fused", "make", "host", "tune", "rebin"):
        px = case["n_q"] * _mean_pixels(case)
    if kind in ("fused", "make", "host"):
        # a skewer's stencil tube: two new voxel faces per cell of path, and not more than the box
        record = {"tensor": 28, "gauss7": 8}.get(case.get("layout"), 8)
        faces = {"gauss7": 49}.get(case.get("layout"), 4)
        box = min(record * case["n"] ** 3, px * DR / CELL * 1.25 * faces * record)
        out = {"fused": 4 if case.get("store") else 0, "make": 8, "host": 4}[kind]
        flops = px * (60 + 5 * math.log2(case["n_fft"]) + (2.5 * math.log2(case["n_fft"]) if kind != "make" else 0)
                      + {"gauss7": 4 * 399, "tensor": 110}.get(case.get("layout"), 28))
        return {"bytes": box + px * out + case["n_q"] * 112, "flops": flops}
    if kind == "tune":
        return {"bytes": 8 * px + 96 * case["n_q"], "flops": px * (30 + 2.5 * math.log2(case["n_fft"]))}
    if kind == "rebin":
        return {"bytes": 8 * px + 4 * px / case["rebin"] + 96 * case["n_q"], "flops": px * 20}
    n = case.get("n", 0)
    if kind == "synth":
        vol, boxes = n ** 3, {"planar": 1, "tensor": 7}.get(case["layout"], 2)
        # a transform larger than the cache reads and writes its data in two passes at least
        return {"bytes": vol * 4 * (boxes + 4), "flops": 2.5 * vol * 3 * math.log2(n) * (1 + boxes)}
    if kind == "draw":
        return {"bytes": 12 * n ** 3 + 32 * case["nbar"] * (n * case["cell"]) ** 3, "flops": 80.0 * n ** 3}
    flops = case["n_samples"] * case["epochs"] * 6.0 * mk.MLP_NPARAM
    return {"bytes": case["n_samples"] * 39 * 4 + mk.MLP_NPARAM * 8, "flops": flops}


# ------------------------------------------------------------------ exact: cosmology in numpy, FP64
class _Cosmology:
    GL_X, GL_W = np.polynomial.legendre.leggauss(8)

    def __init__(self):
        self.z = np.arange(0.0, 12.0 + 1e-9, 1.0 / 256)
        self.dc = np.concatenate([[0.0], np.cumsum(self._quad(self._inv_e, self.z[:-1], self.z[1:]))]) * C_H0
        tail_x, tail_w = np.polynomial.legendre.leggauss(64)  # growth beyond z = 12, in sqrt(a)
        t1 = math.sqrt(1.0 / 13.0)
        t = 0.5 * t1 * (tail_x + 1.0)
        tail = np.sum(0.5 * t1 * tail_w * 2.0 * t ** 4 / (OMEGA_M + (1 - OMEGA_M) * t ** 6) ** 1.5)
        s = self._quad(self._heath, self.z[:-1], self.z[1:])
        self.up = np.concatenate([tail + np.cumsum(s[::-1])[::-1], [tail]])
        self.g0 = self.up[0]

    @staticmethod
    def e(z):
        return np.sqrt(OMEGA_M * (1 + z) ** 3 + 1 - OMEGA_M)

    def _inv_e(self, z):
        return 1.0 / self.e(z)

    def _heath(self, z):
        return (1 + z) / self.e(z) ** 3

    def _quad(self, f, a, b):
        h, m = 0.5 * (b - a), 0.5 * (a + b)
        return sum(w * f(m + h * x) for x, w in zip(self.GL_X, self.GL_W)) * h

    def distance(self, z):
        i = np.clip((z * 256).astype(np.int64), 0, len(self.z) - 1)
        return self.dc[i] + C_H0 * self._quad(self._inv_e, self.z[i], z)

    def redshift(self, r):
        z = np.interp(r, self.dc, self.z)
        for _ in range(4):
            z = z - (self.distance(z) - r) * self.e(z) / C_H0
        return z

    def growth(self, z):
        i = np.clip((z * 256).astype(np.int64), 0, len(self.z) - 1)
        return self.e(z) * (self.up[i] - self._quad(self._heath, self.z[i], z)) / self.g0


class _Pixels:
    """Pixel ranges of a catalogue and the per-pixel tables, in FP64."""

    def __init__(self, w, pos):
        cos = _Cosmology()
        r = np.linalg.norm(pos.cpu().numpy(), axis=1)
        zq = cos.redshift(r)
        z_lo, z_hi = (1 + zq) * w["lrf_min"] / LAMBDA_LYA - 1, (1 + zq) * w["lrf_max"] / LAMBDA_LYA - 1
        if w["lobs_min"] > 0:
            z_lo = np.maximum(z_lo, w["lobs_min"] / LAMBDA_LYA - 1)
        z_lo = np.maximum(z_lo, 0.0)
        j0 = np.ceil(cos.distance(z_lo) / w["dr"] - 0.5).astype(np.int64)
        j1 = np.ceil(cos.distance(np.maximum(z_hi, 0.0)) / w["dr"] - 0.5).astype(np.int64)
        n = np.where((z_hi > z_lo) & (j1 > j0), j1 - j0, 0)
        if w["n_max"] > 0:
            j0 = np.where(n > w["n_max"], j1 - w["n_max"], j0)
            n = np.minimum(n, w["n_max"])
        n = np.where(n < w["n_min"], 0, n)
        self.j0, self.n = torch.from_numpy(j0).cuda(), torch.from_numpy(n).cuda()
        zj = cos.redshift((np.arange(int(j1.max()) + 4096) + 0.5) * w["dr"])
        cum = np.concatenate([[0.0], np.cumsum(zj)])
        nodes = np.asarray(w["node_z"])
        d = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).cuda()  # noqa: E731
        self.growth, self.a = d(cos.growth(zj)), d(np.exp(np.interp(zj, nodes, w["node_ln_a"])))
        self.b, self.c = d(np.interp(zj, nodes, w["node_b"])), d(np.interp(zj, nodes, w["node_c"]))
        self.cum, self.w = d(cum), w

    def zbin(self, j, span):
        """z bin of the mean z of pixels j .. j + span - 1."""
        z = (self.cum[j + span] - self.cum[j]) / span
        f = torch.floor((z - self.w["z_bin_lo"]) / self.w["dz_bin"])
        return f.clamp(-1, self.w["n_zbins"]).long()


def _mul32(m, x):
    """(high, low) words of the 64-bit product of a constant and 32-bit values held in int64."""
    lo, hi = m * (x & 0xFFFF), m * (x >> 16)
    low = (lo + ((hi & 0xFFFF) << 16))
    return ((hi + (lo >> 16)) >> 16), low & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011), words as int64."""
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c0)
        h1, l1 = _mul32(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _unit(x):
    return (x.double() + 0.5) * 2.0 ** -32


def _small_scale(w, ids, seg, z_mean):
    """delta_S of segments (rows): the inverse real DFT of the Philox modes."""
    n, m = w["n_fft"], w["n_fft"] // 2
    c = torch.arange(n // 4, device="cuda")[None, :]
    zero = torch.zeros_like(c)
    x, y, z, t = _philox(c + 0 * seg[:, None], seg[:, None] + zero, (ids >> 32)[:, None] + zero, zero + 0 * seg[:, None],
                         torch.full_like(c, w["seed_noise"]), (ids & 0xFFFFFFFF)[:, None])
    p = torch.as_tensor(np.asarray(w["p_s"]), device="cuda").reshape(-1, m + 1)
    if len(p) > 1:
        zs = torch.as_tensor(np.asarray(w["p_s_z"]), device="cuda")
        i = (torch.searchsorted(zs, z_mean, right=True) - 1).clamp(0, len(p) - 2)
        f = ((z_mean - zs[i]) / (zs[i + 1] - zs[i])).clamp(0, 1)[:, None]
        p = p[i] * (1 - f) + p[i + 1] * f
    amp = torch.sqrt(n * p / w["dr"])
    modes = torch.zeros((len(seg), m + 1), dtype=torch.complex128, device="cuda")
    r0, r1 = torch.sqrt(-torch.log(_unit(x))), torch.sqrt(-torch.log(_unit(z)))
    a0, a1 = 2 * math.pi * _unit(y), 2 * math.pi * _unit(t)
    modes[:, 0:m:2] = torch.polar(r0, a0)
    modes[:, 1:m:2] = torch.polar(r1, a1)
    modes[:, m] = math.sqrt(2.0) * r0[:, 0] * torch.cos(a0[:, 0])
    modes[:, 0] = 0
    return torch.fft.irfft(modes * amp, n=n)


def _corner(box, ix, iy, iz, n):
    return box.reshape(-1)[((iz % n) * n + iy % n) * n + ix % n].double()


def _interpolate(case, boxes, at):
    """(delta, eta fields...) at cell coordinates `at` (voxel centres at integers)."""
    n = case["n"]
    if case.get("layout") == "gauss7":
        c = torch.floor(at + 0.5).long()
        o = torch.arange(-3, 4, device="cuda")
        wt = torch.exp(-0.5 * (c[..., None] + o - at[..., None]) ** 2)
        wt = wt / wt.sum(-1, keepdim=True)
        got = [torch.zeros(at.shape[:-1], dtype=torch.float64, device="cuda") for _ in boxes]
        for k in range(7):
            for j in range(7):
                wkj = wt[:, 2, k] * wt[:, 1, j]
                row = (((c[:, 2] + k - 3) % n) * n + (c[:, 1] + j - 3) % n) * n
                for i in range(7):
                    v, idx = wkj * wt[:, 0, i], row + (c[:, 0] + i - 3) % n
                    for g, b in zip(got, boxes):
                        g += v * b.reshape(-1)[idx]
        return got
    c = torch.floor(at).long()
    f = at - c
    got = []
    for b in boxes:
        v = torch.zeros(at.shape[:-1], dtype=torch.float64, device="cuda")
        for q in range(8):
            dx, dy, dz = q & 1, (q >> 1) & 1, q >> 2
            wt = (f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (f[:, 2] if dz else 1 - f[:, 2])
            v += wt * _corner(b, c[:, 0] + dx, c[:, 1] + dy, c[:, 2] + dz, n)
        got.append(v)
    return got


class _Sums:
    """Statistics over rows of segments, per z bin."""

    def __init__(self, w, rebin, tables):
        self.w, self.rebin, self.t = w, rebin, tables
        self.s = torch.zeros((w["n_zbins"], 10), dtype=torch.float64, device="cuda")
        self.p = torch.zeros((w["n_zbins"], w["n_kbins"]), dtype=torch.float64, device="cuda")
        self.g = torch.zeros(w["n_zbins"], dtype=torch.float64, device="cuda")

    def add(self, j, valid, f, d, e):
        """j: first fine pixel of every value; rows are segments of n_fft values, `valid` those that exist."""
        w, n, r = self.w, self.w["n_fft_p1d"], self.rebin
        zb = torch.where(valid, self.t.zbin(j, r), -1)
        for b in range(w["n_zbins"]):
            m = zb == b
            if not bool(m.any()):
                continue
            F, D, E = f[m], d[m], e[m]
            q = [torch.ones_like(F), F, F * F, D, E, D * D, E * E, D * E, F * D, F * E]
            self.s[b] += torch.stack([v.sum() for v in q])
        full = valid[:, -1]
        x = torch.fft.rfft(f[full])[:, 1:]
        power = (x.real ** 2 + x.imag ** 2) * (r * w["dr"] / n)
        power = power.reshape(len(power), w["n_kbins"], -1).sum(-1)
        zs = self.t.zbin(j[full, 0], n * r)
        for b in range(w["n_zbins"]):
            self.p[b] += power[zs == b].sum(0)
            self.g[b] += (zs == b).sum()

    def result(self):
        w = self.w
        s, p, g = self.s.cpu().numpy(), self.p.cpu().numpy(), self.g.cpu().numpy()
        out = dict(sums=s, n_seg=g, p1d_df=np.zeros_like(p), **{k: np.zeros(len(s)) for k in
                   ("mean_flux", "sigma_f", "b_f", "beta_f")})
        for b in range(len(s)):
            if s[b, 0] <= 0:
                continue
            m = s[b, 1:] / s[b, 0]
            out["mean_flux"][b] = m[0]
            out["sigma_f"][b] = math.sqrt(max(m[1] - m[0] ** 2, 0.0))
            cdd, cee, cde = m[4] - m[2] ** 2, m[5] - m[3] ** 2, m[6] - m[2] * m[3]
            vd, ve = m[7] - m[0] * m[2], m[8] - m[0] * m[3]
            det = cdd * cee - cde ** 2
            if det != 0:
                kd, ke = (cee * vd - cde * ve) / det, (cdd * ve - cde * vd) / det
                out["b_f"][b], out["beta_f"][b] = kd / m[0], ke / kd if kd else 0.0
            if g[b] > 0:
                out["p1d_df"][b] = p[b] / (g[b] * (w["n_fft_p1d"] // 2 // w["n_kbins"])) / m[0] ** 2
        thick = s[:, 0] >= THIN
        r = {"pixels": None, "segments": None, "sums": s[:, 1:], "p1d": out["p1d_df"], "mean_flux": out["mean_flux"]}
        r.update({k: np.where(thick, out[k], 0.0) for k in ("sigma_f", "b_f", "beta_f")})
        return r


def _segments(n_out, size):
    """(skewer, segment number) of every segment of `size` values, in order."""
    per = (n_out + size - 1) // size
    sk = torch.repeat_interleave(torch.arange(len(n_out), device="cuda"), per)
    first = torch.cumsum(per, 0) - per
    return sk, torch.arange(len(sk), device="cuda") - first[sk]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("draw", "train"):  # decisions and 16-bit training steps have no 64-bit value
        return None
    if kind == "synth":
        return _exact_synth(case, seed)
    w = _recipe(case, seed)
    pos, ids = _catalogue(case, seed)
    t = _Pixels(w, pos)
    total = int(t.n.sum())
    start = torch.cumsum(t.n, 0) - t.n
    rebin = case.get("rebin", 1)
    n_out = t.n // rebin
    out0 = torch.cumsum(n_out, 0) - n_out
    stored = kind in ("tune", "rebin")
    if stored:
        fd, fe = _stored_fields(total, seed)
    else:
        delta, eta = _box(case["n"], seed, SIX if case.get("layout") == "tensor" else XX)
        boxes = [delta] + eta
        u = pos / pos.norm(dim=1, keepdim=True)
        origin = torch.tensor(w["origin"], device="cuda", dtype=torch.float64)
    want = 2 if kind == "make" else 1
    flux = [torch.empty(int(n_out.sum()), dtype=torch.float64, device="cuda") for _ in range(want)]
    sums = _Sums(w, rebin, t)
    n = w["n_fft"]
    sk, seg = _segments(n_out, n)
    rows = max(1, (1 << (22 if case.get("layout") == "gauss7" else 24)) // n)
    for a in range(0, len(sk), rows):
        s, g = sk[a:a + rows], seg[a:a + rows]
        p = g[:, None] * n + torch.arange(n, device="cuda")[None, :]
        valid = p < n_out[s][:, None]
        j = t.j0[s][:, None] + p * rebin
        if stored:
            at = torch.where(valid, start[s][:, None] + p * rebin, 0)
            D = E = F = 0.0
            for r in range(rebin):
                d, e = fd[at + r].double(), fe[at + r].double()
                D, E, F = D + d, E + e, F + torch.exp(-t.a[j + r] * torch.exp(t.b[j + r] * (d + t.c[j + r] * e)))
            D, E, F = D / rebin, E / rebin, F / rebin
        else:
            z = (t.cum[j[:, 0] + n] - t.cum[j[:, 0]]) / n
            ds = _small_scale(w, ids[s], g, z)
            v = valid.reshape(-1)
            x = (((j.double() + 0.5) * w["dr"])[..., None] * u[s][:, None, :] - origin) / w["cell"] - 0.5
            got = _interpolate(case, boxes, x.reshape(-1, 3)[v])
            if len(got) > 2:
                q = u[s][:, None, :].expand(-1, n, -1).reshape(-1, 3)[v]
                got = [got[0], sum((1 if i == k else 2) * q[:, i] * q[:, k] * f for (i, k), f in zip(SIX, got[1:]))]
            D, E = torch.zeros_like(ds), torch.zeros_like(ds)
            D[valid], E[valid] = got[0], got[1]
            D, E = t.growth[j] * D + ds, t.growth[j] * E
            F = torch.exp(-t.a[j] * torch.exp(t.b[j] * (D + t.c[j] * E)))
        o = (out0[s][:, None] + p)[valid]
        if kind == "make":
            flux[0][o], flux[1][o] = D[valid], E[valid]
        else:
            flux[0][o] = F[valid]
            sums.add(j, valid, torch.where(valid, F, 0.0), D, E)
    if kind == "make":
        return {"sk": None, "offsets": None, "delta": flux[0], "eta": flux[1]}
    r = sums.result()
    if kind == "rebin" or kind == "host" or case.get("store"):
        r["flux"] = flux[0]
    return r


def _exact_synth(case, seed):
    n, cell = case["n"], case["cell"]
    noise = torch.empty(n ** 3, dtype=torch.float64, device="cuda")
    step = 1 << 24
    for a in range(0, n ** 3 // 4, step):
        c = torch.arange(a, min(a + step, n ** 3 // 4), device="cuda")
        z = torch.zeros_like(c)
        x, y, p, q = _philox(c & 0xFFFFFFFF, c >> 32, z, z, z + (seed & 0xFFFFFFFF), z + (seed >> 32))
        r0, r1 = torch.sqrt(-2 * torch.log(_unit(x))), torch.sqrt(-2 * torch.log(_unit(p)))
        a0, a1 = 2 * math.pi * _unit(y), 2 * math.pi * _unit(q)
        v = torch.stack([r0 * torch.cos(a0), r0 * torch.sin(a0), r1 * torch.cos(a1), r1 * torch.sin(a1)], 1)
        noise[4 * a:4 * a + v.numel()] = v.reshape(-1)
    f = torch.fft.rfftn(noise.reshape(n, n, n))
    del noise
    pk, dk = _pk_table(cell)
    table = torch.from_numpy(pk).cuda()
    m = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * (2 * math.pi / (n * cell))
    kx, ky = m[: n // 2 + 1].abs(), m
    for iz in range(n):
        k2 = kx[None, :] ** 2 + ky[:, None] ** 2 + ky[iz] ** 2
        u = torch.sqrt(k2) / dk
        i = u.long().clamp(0, len(pk) - 2)
        p = torch.where(u <= len(pk) - 1, table[i] + (u - i) * (table[i + 1] - table[i]), 0.0)
        p[:, n // 2] = 0
        p[n // 2, :] = 0
        p[k2 == 0] = 0
        f[iz] *= torch.sqrt(p.clamp_min(0) / cell ** 3) * (iz != n // 2)
    margin, layout = {"planar": 0, "halo": 3}.get(case["layout"], 0), case["layout"]
    size = {"planar": n, "halo": n + 6}.get(layout, n + 1)
    at = (torch.arange(size, device="cuda") - margin) % n

    def spread(b):
        return b[at][:, at][:, :, at]

    fields = {"planar": [], "tensor": SIX}.get(layout, XX)
    width = {"planar": 1, "tensor": 8}.get(layout, 2)
    out = torch.zeros((size, size, size, width), dtype=torch.float64, device="cuda")
    out[..., 0] = spread(torch.fft.irfftn(f, s=(n, n, n)))
    for s, (a, b) in enumerate(fields):
        g = f.clone()
        for iz in range(n):
            ks = (m[None, : n // 2 + 1], m[:, None], m[iz])
            k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
            g[iz] *= -ks[a] * ks[b] / torch.where(k2 > 0, k2, torch.ones_like(k2))
        out[..., 1 + s] = spread(torch.fft.irfftn(g, s=(n, n, n)))
        del g
    return out.reshape(-1)
