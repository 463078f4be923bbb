"""The workloads by which the imager's speed is judged.

A case is one call, or one short sequence of calls, that a program using the package makes
over and over: image a set of visibilities, differentiate an image, predict visibilities
from an image, take a training step of the gridding kernel, evaluate the direct transform.
``listed()`` holds the sizes the package is used at, ``draw(rng)`` gives further ones of the
same ranges, ``prepare``/``run`` are one pass of a case, ``work`` the bytes and operations a
pass cannot do without, ``exact`` its outputs in 64 bits from plain torch.

Inputs are synthetic observations: earth-rotation tracks of a random station layout
(core-dense, uneven coverage) or a uniform disk of (u, v); values of a few point sources
plus noise.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_2301_06061_gb300 import autograd, wst

DEV = "cuda"
LEARNED_TABLE = os.path.join(os.path.dirname(os.path.abspath(wst.__file__)), "data", "learned_kernel_w8.npz")
C_LIGHT = 299_792_458.0
DIAMETER_M = 20_000.0  # of the station layout
FREQ_HZ = (120e6, 168e6)
LATITUDE_DEG, DECLINATION_DEG, TRACK_HOURS = 52.9, 45.0, 8.0
KB_PER_CELL = 128
CHUNK = 1 << 23  # visibilities per step of the input generator

# what: "image"      bind the visibilities and image them
#       "staged"     bind, then the gridder, the transform and the correction by their own calls
#       "grad"       the image and its gradient by the values
#       "degrid"     visibilities predicted from an image, the coordinates bound before
#       "table_grad" the image and its gradient by the samples of a tabulated kernel
#       "direct"     Eq. 1 for a point sky, then the direct transform at chosen pixels
# w_half: half the w range of the plan (0: from the data); fold, chunk: plan options
DEFAULTS = {
    "what": "image", "n": 256, "grid_n": 0, "fov": 0.1, "n_w": 8, "n_vis": 10_000, "batch": 1, "w_half": 0.0,
    "support": 7, "kernel": "gauss", "cover": "tracks", "stations": 60, "channels": 16, "rows": False,
    "weights": False, "fold": False, "chunk": 0, "sources": 6, "pixels": 0,
}


def _case(**kw) -> dict:
    return dict(DEFAULTS, **kw)


def listed() -> list[dict]:
    return [
        # a quick look at one short observation: launches and latency are all there is
        _case(name="tiny_image", n=256, fov=0.1, n_w=8, n_vis=10_000, cover="disk", w_half=200.0),
        # an array's 8 h observation as it is recorded, by baseline row and channel
        _case(name="array_rows", n=4096, fov=0.2, n_w=32, n_vis=4_078_080, rows=True),
        # the wide-field survey image: the benchmark's size
        _case(name="wide_field", n=16384, fov=0.5, n_w=32, n_vis=100_000_000, stations=300, channels=64),
        # a spectral cube: one image per channel with uneven counts, in one call
        _case(name="channel_cube", n=2048, fov=0.09, n_w=16, n_vis=37_700_000, batch=64, channels=1),
        # a wide field with the learned kernel and imaging weights
        _case(name="table_weighted", n=8192, fov=0.25, n_w=16, n_vis=20_000_000, stations=150, channels=32,
              support=8, kernel="learned", weights=True),
        # a padded grid (factor 1.25) against edge aliasing; odd plane and visibility counts
        _case(name="padded_es", n=3276, grid_n=4096, fov=0.16, n_w=21, n_vis=1_234_567, support=8, kernel="es"),
        # a large image under a memory limit: planes streamed eight at a time, w folded
        _case(name="streamed_fold", n=16384, fov=0.5, n_w=16, n_vis=20_000_000, stations=300, channels=64, rows=True,
              fold=True, chunk=8),
        # the gridder, the transform and the correction as separate calls, a shorter kernel
        _case(name="staged_calls", what="staged", n=1024, fov=0.03125, n_w=12, n_vis=300_001, support=6),
        # deconvolution or calibration by gradient: the image and its gradient by the values
        _case(name="image_grad", what="grad", n=2048, fov=0.09, n_w=16, n_vis=1_000_000, channels=1),
        # a major cycle's prediction: a model image degridded at every visibility
        _case(name="predict_image", what="degrid", n=8192, fov=0.25, n_w=16, n_vis=10_000_000, stations=150,
              channels=32),
        # a training step of the learned kernel: image and table gradient of one sky
        _case(name="train_step", what="table_grad", n=512, fov=0.1, n_w=8, n_vis=200_000, support=8, kernel="learned",
              cover="disk", w_half=200.0),
        # that step's data: Eq. 1 for the sky, the direct transform at the sampled pixels
        _case(name="train_data", what="direct", n=512, fov=0.1, n_w=8, n_vis=200_000, cover="disk", w_half=200.0,
              sources=25, pixels=2048),
    ]


def _log_int(rng, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    what = rng.choice(["image"] * 8 + ["staged", "grad", "grad", "degrid", "degrid", "table_grad", "direct"])
    if what == "direct":
        n_vis = _log_int(rng, 2e3, 2e6)
        pixels = max(1, min(_log_int(rng, 16, 4096), int(8e8 / n_vis)))
        n = rng.choice([256, 512, 1000, 4096])
        return _case(what=what, n=n, n_vis=n_vis, fov=rng.uniform(0.05, 0.3), cover="disk",
                     w_half=rng.uniform(50.0, 400.0), sources=rng.randint(1, 50), pixels=pixels)
    log_m = {"image": (8, 14), "staged": (8, 12), "grad": (8, 12), "degrid": (9, 14), "table_grad": (8, 11)}[what]
    m = 1 << rng.randint(*log_m)
    batch = 1
    if what == "image" and m <= 2048 and rng.random() < 0.4:
        batch = rng.randint(2, 48)
    n_w = _log_int(rng, 4, 40)
    budget = (16384 ** 2 * 32) // 2  # cells of all planes, half of the largest listed case
    n_w = max(1, min(n_w, budget // (m * m * batch)))
    cells = m * m * batch
    n_vis = _log_int(rng, max(1000.0, 0.02 * cells), min(5e7, 1.0 * cells + 1000.0))
    # padded grids: the image an even number of pixels, the grid a power of two above it
    n, grid_n = m, 0
    if rng.random() < 0.3:
        n, grid_n = 2 * rng.randint(m // 4 + 1, m // 2 - 1), m
    extent = rng.uniform(10_500.0, 16_384.0)  # wavelengths from the grid's centre to its edge
    support = rng.choice([7, 7, 7, 8, 8, 8, 5, 6, 9, 10])
    kernel = rng.choice(["gauss", "gauss", "gauss", "es", "kb"] + (["learned"] if support == 8 else []))
    if what == "table_grad":
        support, kernel = 8, rng.choice(["learned", "kb"])
    disk = m <= 512 and rng.random() < 0.5
    return _case(
        what=what, n=n, grid_n=grid_n, fov=n / (2.0 * extent), n_w=n_w, n_vis=n_vis, batch=batch, support=support,
        kernel=kernel, cover="disk" if disk else "tracks", w_half=rng.uniform(100.0, 400.0) if disk else 0.0,
        stations=rng.choice([60, 150, 300]) if n_vis > 1_000_000 else 60,
        channels=1 if batch > 1 else rng.choice([1, 16, 32, 64]),
        rows=what == "image" and batch == 1 and not disk and rng.random() < 0.4,
        weights=rng.random() < 0.4, fold=what == "image" and kernel in ("gauss", "es") and rng.random() < 0.25,
        chunk=rng.randint(1, n_w) if rng.random() < 0.2 else 0)


# ----------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------

def _counts(case: dict) -> list[int]:
    """Visibilities of each image: spread over a factor of twenty, the same for every seed."""
    b, total = case["batch"], case["n_vis"]
    if b == 1:
        return [total]
    share = 20.0 ** np.random.default_rng([b, total]).random(b)
    counts = [int(x) for x in np.floor(total * share / share.sum())]
    counts[-1] += total - sum(counts)
    return counts


def _baselines(stations: int, rng) -> torch.Tensor:
    """Equatorial baseline vectors (metres) of stations uniform in a disk, FP64 [pairs, 3]."""
    r = 0.5 * DIAMETER_M * np.sqrt(rng.random(stations))
    th = 2.0 * np.pi * rng.random(stations)
    east, north = r * np.cos(th), r * np.sin(th)
    lat = math.radians(LATITUDE_DEG)
    xyz = np.stack([-math.sin(lat) * north, east, math.cos(lat) * north], axis=1)
    i, j = np.triu_indices(stations, k=1)
    return torch.from_numpy(xyz[j] - xyz[i]).to(DEV)


def _tracks(bl: torch.Tensor, dumps: int) -> torch.Tensor:
    """(u, v, w) in metres over the track, ordered (time, baseline), FP64 [rows, 3]."""
    dec = math.radians(DECLINATION_DEG)
    h = torch.linspace(-0.5, 0.5, dumps, dtype=torch.float64, device=DEV)[:, None] * (TRACK_HOURS * math.pi / 12.0)
    lx, ly, lz = bl[None, :, 0], bl[None, :, 1], bl[None, :, 2]
    s, c = torch.sin(h), torch.cos(h)
    u = s * lx + c * ly
    v = math.sin(dec) * (s * ly - c * lx) + math.cos(dec) * lz
    w = math.cos(dec) * (c * lx - s * ly) + math.sin(dec) * lz
    return torch.stack([u, v, w], dim=-1).reshape(-1, 3).contiguous()


def _expand(rows: torch.Tensor, scale: torch.Tensor, n_vis: int):
    return [torch.outer(rows[:, k], scale).reshape(-1)[:n_vis].float().contiguous() for k in range(3)]


def _values(u, v, w, l, m, flux, gen) -> torch.Tensor:
    """Eq. 1 for a few point sources (phases in 64 bits) plus noise, complex64."""
    out = torch.empty(u.numel(), dtype=torch.complex64, device=DEV)
    for a in range(0, u.numel(), CHUNK):
        ud, vd, wd = (x[a:a + CHUNK].double() for x in (u, v, w))
        acc = torch.view_as_real(out[a:a + CHUNK])
        acc.normal_(0.0, 0.05, generator=gen)
        for ls, ms, fs in zip(l, m, flux):
            ns = -(ls * ls + ms * ms) / (1.0 + math.sqrt(1.0 - ls * ls - ms * ms))
            ph = ud * ls + vd * ms + wd * ns
            ph = (ph - ph.round()).float() * (-2.0 * math.pi)
            acc[:, 0] += fs * torch.cos(ph)
            acc[:, 1] += fs * torch.sin(ph)
    return out


def _table(case: dict):
    """FP32 samples of the case's tabulated kernel on [-W/2, W/2], or None."""
    if case["kernel"] == "learned":
        with np.load(LEARNED_TABLE) as f:
            return f["table"].astype(np.float32)
    if case["kernel"] == "kb":  # Kaiser-Bessel
        W = case["support"]
        beta = math.pi * math.sqrt((0.5 * W) ** 2 - 0.8)
        x = np.linspace(-1.0, 1.0, W * KB_PER_CELL + 1)
        return (np.i0(beta * np.sqrt(np.clip(1.0 - x * x, 0.0, None))) / np.i0(beta)).astype(np.float32)
    return None


def _kparam(case: dict) -> float:
    """sigma of the Gaussian (the package's defaults at 7 and 8), beta of the ES kernel."""
    W = case["support"]
    return 2.3 * W if case["kernel"] == "es" else {7: 0.875, 8: 0.925}.get(W, 0.875 * math.sqrt(W / 7.0))


def _inputs(case: dict, seed: int) -> dict:
    rng = np.random.default_rng([int(seed), 101])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    n, fov, n_vis = case["n"], case["fov"], case["n_vis"]
    d = {"rows": None, "scale": None, "offsets": None, "weight": None}
    if case["cover"] == "disk":
        rad, th, wr = (torch.rand(n_vis, generator=gen, device=DEV, dtype=torch.float64) for _ in range(3))
        rad = 0.45 * n / fov * rad.sqrt()
        th = 2.0 * math.pi * th
        d["u"], d["v"] = (rad * torch.cos(th)).float(), (rad * torch.sin(th)).float()
        d["w"] = ((2.0 * wr - 1.0) * case["w_half"]).float()
        if case["batch"] > 1:
            d["offsets"] = [0] + [int(x) for x in np.cumsum(_counts(case))]
    else:
        bl = _baselines(case["stations"], rng)
        if case["batch"] > 1:  # one channel's tracks per image
            freqs, parts = np.linspace(*FREQ_HZ, case["batch"]), []
            for f, cnt in zip(freqs, _counts(case)):
                rows = _tracks(bl, max(2, -(-cnt // bl.shape[0])))[:cnt]
                parts.append((rows * (f / C_LIGHT)).float())
            uvw = torch.cat(parts)
            d["u"], d["v"], d["w"] = (uvw[:, k].contiguous() for k in range(3))
            d["offsets"] = [0] + [int(x) for x in np.cumsum(_counts(case))]
        else:
            ch = case["channels"]
            d["scale"] = torch.linspace(*FREQ_HZ, ch, dtype=torch.float64, device=DEV) / C_LIGHT
            d["rows"] = _tracks(bl, max(2, -(-n_vis // (bl.shape[0] * ch))))
            d["u"], d["v"], d["w"] = _expand(d["rows"], d["scale"], n_vis)
    k = case["sources"]
    d["l"], d["m"] = rng.uniform(-0.4 * fov, 0.4 * fov, k), rng.uniform(-0.4 * fov, 0.4 * fov, k)
    d["flux"] = 1.0 / (100.0 - 99.0 * rng.random(k))  # dN/dS ~ S^-2 on [0.01, 1]
    if case["what"] == "direct":
        d["pa"] = torch.randint(0, n, (case["pixels"],), generator=gen, device=DEV, dtype=torch.int32)
        d["pb"] = torch.randint(0, n, (case["pixels"],), generator=gen, device=DEV, dtype=torch.int32)
    else:
        d["vis"] = _values(d["u"], d["v"], d["w"], d["l"], d["m"], d["flux"], gen)
    if case["weights"]:
        d["weight"] = torch.rand(n_vis, generator=gen, device=DEV) * 1.5 + 0.25
    if case["what"] in ("grad", "degrid", "table_grad"):  # a residual or model image
        x = torch.randn((case["batch"], n, n, 2), generator=gen, device=DEV)
        d["dimage"] = torch.view_as_complex(x)
    return d


# ----------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------

def prepare(case: dict, seed: int) -> dict:
    st = dict(_inputs(case, seed), case=case)
    if case["what"] == "direct":
        for k in ("l", "m", "flux"):
            st[k] = torch.from_numpy(np.ascontiguousarray(st[k])).to(DEV)
        return st
    table = _table(case)
    kind = {"gauss": wst.WST_KERNEL_GAUSS, "es": wst.WST_KERNEL_ES}.get(case["kernel"], wst.WST_KERNEL_TABLE)
    wh = case["w_half"]
    cfg = wst.Config(n=case["n"], fov=case["fov"], n_w=case["n_w"], w_min=-wh, w_max=wh, support=case["support"],
                     kernel=kind, kparam=_kparam(case), ktable_len=0 if table is None else int(table.size),
                     flags=wst.WST_FLAG_KAHAN | (wst.WST_FLAG_WFOLD if case["fold"] else 0),
                     planes_per_chunk=case["chunk"], batch=case["batch"], grid_n=case["grid_n"])
    if case["fold"] and wh > 0.0:
        cfg.w_min = 0.0
    plan = st["plan"] = wst.Plan(cfg)
    if table is not None:
        st["table"] = torch.from_numpy(table).to(DEV)
        if case["what"] != "table_grad":
            plan.set_kernel_table(st["table"])
    plan.ensure_workspace(case["n_vis"])
    if case["what"] == "degrid":
        plan.set_vis(st["u"], st["v"], st["w"], st["vis"], st["weight"])
    return st


def run(st: dict):
    case, what = st["case"], st["case"]["what"]
    if what == "direct":
        vis = torch.empty(case["n_vis"], dtype=torch.complex64, device=DEV)
        wst.wst_predict_points(st["u"], st["v"], st["w"], st["l"], st["m"], st["flux"], vis)
        out = torch.empty(case["pixels"], dtype=torch.complex64, device=DEV)
        wst.wst_dft(st["u"], st["v"], st["w"], vis, case["n"], case["fov"], st["pa"], st["pb"], out, st["weight"])
        return vis, out
    plan = st["plan"]
    if what == "degrid":
        return plan.degrid(st["dimage"])
    if what == "grad":
        vis = st["vis"].detach().requires_grad_()
        img = autograd.image(vis, plan, st["u"], st["v"], st["w"], st["weight"])
        return img.detach(), torch.autograd.grad(img, vis, st["dimage"])[0]
    if what == "table_grad":
        table = st["table"].detach().requires_grad_()
        img = autograd.kernel_image(table, plan, st["u"], st["v"], st["w"], st["vis"], st["weight"])
        return img.detach(), torch.autograd.grad(img, table, st["dimage"])[0]
    if case["rows"]:
        plan.set_vis_rows(st["rows"], st["scale"], st["vis"], st["weight"], st["offsets"])
    else:
        plan.set_vis(st["u"], st["v"], st["w"], st["vis"], st["weight"], st["offsets"])
    if what == "image":
        return plan.image()
    m, planes = case["grid_n"] or case["n"], case["n_w"]
    grid = torch.empty((planes, m, m), dtype=torch.complex64, device=DEV)
    img = torch.zeros((1, case["n"], case["n"]), dtype=torch.complex64, device=DEV)
    wst.wst_grid(plan.handle, 0, planes, grid)
    wst.wst_fft_correct(plan.handle, 0, planes, grid, img)
    wst.wst_correct(plan.handle, img)
    return img


def work(case: dict) -> dict:
    """Every input read once, every output written once; the taps, transforms and screens."""
    n_vis, n, m = case["n_vis"], case["n"], case["grid_n"] or case["n"]
    weight = 4 * n_vis if case["weights"] else 0
    if case["what"] == "direct":
        pairs = n_vis * (case["sources"] + case["pixels"])
        return {"bytes": 20 * n_vis + weight + 8 * n_vis + 16 * case["pixels"], "flops": 24.0 * pairs}
    if case["rows"]:
        coords = 24 * -(-n_vis // case["channels"]) + 8 * case["channels"]
    else:
        coords = 12 * n_vis
    image = 8 * n * n * case["batch"]
    planes = case["n_w"] * case["batch"]
    one_way = (4.0 * case["support"] ** 2 * n_vis + planes * (10.0 * m * m * math.log2(m) + 8.0 * n * n))
    if case["what"] == "degrid":
        return {"bytes": coords + weight + image + 8 * n_vis, "flops": one_way}
    bytes_, flops = coords + weight + 8 * n_vis + image, one_way
    if case["what"] in ("grad", "table_grad"):
        bytes_ += image + (8 * n_vis if case["what"] == "grad" else 8 * 8193)
        flops *= 2.0
    return {"bytes": bytes_, "flops": flops}


# ----------------------------------------------------------------------------------------
# the same outputs in 64 bits
# ----------------------------------------------------------------------------------------

class _Kernel:
    def __init__(self, case: dict):
        self.W, self.kind, self.param = case["support"], case["kernel"], _kparam(case)
        t = _table(case)
        self.t = None if t is None else torch.from_numpy(t).to(DEV).double()

    def _position(self, x):
        """Table interval and fraction of the arguments x."""
        pos = (x + 0.5 * self.W) * ((self.t.numel() - 1) / self.W)
        i = pos.floor().long().clamp_(0, self.t.numel() - 2)
        return i, pos - i

    def __call__(self, x):
        if self.t is not None:
            i, f = self._position(x)
            return self.t[i] * (1.0 - f) + self.t[i + 1] * f
        if self.kind == "es":
            z = 2.0 * x / self.W
            return torch.exp(self.param * (torch.sqrt((1.0 - z * z).clamp_(min=0.0)) - 1.0))
        return torch.exp(-x * x / (2.0 * self.param ** 2))

    def spread(self, out, x, val):
        """out += d(sum val G(x)) / d(table)."""
        i, f = self._position(x)
        out.index_add_(0, i, val * (1.0 - f))
        out.index_add_(0, i + 1, val * f)

    def transform(self, m: int):
        """Ghat(nu_a), nu_a = (a - m/2)/m: Gauss-Legendre panels over the support."""
        panels = 64 * self.W if self.t is None else self.t.numel() - 1
        gx, gw = np.polynomial.legendre.leggauss(8 if self.t is None else 4)
        h = self.W / panels
        x = (-0.5 * self.W + h * (np.arange(panels)[:, None] + 0.5 * (gx + 1.0))).ravel()
        x = torch.from_numpy(x).to(DEV)
        g = self(x) * torch.from_numpy(np.tile(0.5 * h * gw, panels)).to(DEV)
        nu = (torch.arange(m, device=DEV, dtype=torch.float64) - m // 2) / m
        step = max(1, (1 << 26) // x.numel())
        return torch.cat([torch.cos(2.0 * math.pi * nu[a:a + step, None] * x) @ g for a in range(0, m, step)])


class _Geometry:
    """One image's visibilities, placed on the cells and planes of its grid."""

    def __init__(self, case: dict, u, v, w, vis, weight, kernel: _Kernel):
        m, n, self.W = case["grid_n"] or case["n"], case["n"], case["support"]
        self.m, self.n, self.n_w, self.k = m, n, case["n_w"], kernel
        fov = case["fov"] * m / n
        if case["fold"]:
            neg = w < 0
            s = torch.where(neg, -1.0, 1.0)
            u, v, w, vis = u * s, v * s, w * s, torch.where(neg, vis.conj(), vis)
        if case["w_half"] > 0.0:
            lo, hi = (0.0 if case["fold"] else -case["w_half"]), case["w_half"]
        else:
            lo, hi = float(w.min()), float(w.max())
        hx = (0.5 * m + u.double() * fov) - 0.5 * self.W
        hy = (0.5 * m + v.double() * fov) - 0.5 * self.W
        i0, j0 = hx.ceil(), hy.ceil()
        kept = ((i0 >= 0) & (j0 >= 0) & (i0 + self.W <= m) & (j0 + self.W <= m)).nonzero().squeeze(1)
        scale = self.n_w / (hi - lo) if hi > lo else 0.0
        plane = ((w.double() - lo) * scale).floor().clamp_(0, self.n_w - 1).long()[kept]
        plane, order = plane.sort()
        self.idx = kept[order]  # visibility of each placed record, plane by plane
        self.gx, self.gy = (i0 - hx)[self.idx], (j0 - hy)[self.idx]
        self.cell = (j0 * m + i0).long()[self.idx]
        val = vis.to(torch.complex128)
        self.wt = torch.ones(len(val), dtype=torch.float64, device=DEV) if weight is None else weight.double()
        self.val = (val * self.wt)[self.idx]
        self.wt = self.wt[self.idx]
        self.begin = [0] + torch.bincount(plane, minlength=self.n_w).cumsum(0).tolist()
        self.wk = [lo + (k + 0.5) * (hi - lo) / self.n_w for k in range(self.n_w)]
        l = (torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) * (case["fov"] / n)
        r2 = l[:, None] ** 2 + l[None, :] ** 2
        self.inside = r2 < 1.0
        self.t = -r2 / (1.0 + torch.sqrt((1.0 - r2).clamp_(min=0.0)))
        self.crop = slice((m - n) // 2, (m - n) // 2 + n)

    def taps(self, k: int):
        """(record range, cell, G_x G_y, tap arguments) of every tap of plane k."""
        for a in range(self.begin[k], self.begin[k + 1], CHUNK):
            s = slice(a, min(a + CHUNK, self.begin[k + 1]))
            xs = [j - 0.5 * self.W + self.gx[s] for j in range(self.W)]
            gxs = [self.k(x) for x in xs]
            for d in range(self.W):
                y = d - 0.5 * self.W + self.gy[s]
                gy = self.k(y)
                for j in range(self.W):
                    yield s, self.cell[s] + (d * self.m + j), gxs[j], gy, xs[j], y

    def screen(self, k: int):
        ph = self.wk[k] * self.t
        ph = (ph - ph.round()) * (2.0 * math.pi)
        return torch.complex(torch.cos(ph), torch.sin(ph)) * self.inside

    def image(self):
        out = torch.zeros((self.n, self.n), dtype=torch.complex128, device=DEV)
        for k in range(self.n_w):
            if self.begin[k] == self.begin[k + 1]:
                continue
            g = torch.zeros((self.m * self.m, 2), dtype=torch.float64, device=DEV)
            for s, cell, gx, gy, _, _ in self.taps(k):
                g.index_add_(0, cell, torch.view_as_real(self.val[s]) * (gx * gy)[:, None])
            g = torch.view_as_complex(g).view(self.m, self.m)
            f = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(g), norm="forward"))
            out += f[self.crop, self.crop] * self.screen(k)
        return out

    def plane_adjoint(self, dimage, k: int):
        x = torch.zeros((self.m, self.m), dtype=torch.complex128, device=DEV)
        x[self.crop, self.crop] = dimage * self.screen(k).conj()
        return torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(x))).reshape(-1)

    def degrid(self, dimage, n_vis: int):
        got = torch.zeros(len(self.idx), dtype=torch.complex128, device=DEV)
        for k in range(self.n_w):
            if self.begin[k] == self.begin[k + 1]:
                continue
            h = self.plane_adjoint(dimage, k)
            for s, cell, gx, gy, _, _ in self.taps(k):
                got[s] += h[cell] * (gx * gy)
        out = torch.zeros(n_vis, dtype=torch.complex128, device=DEV)
        out[self.idx] = got * self.wt
        return out

    def table_grad(self, dimage):
        out = torch.zeros(self.k.t.numel(), dtype=torch.float64, device=DEV)
        for k in range(self.n_w):
            if self.begin[k] == self.begin[k + 1]:
                continue
            h = self.plane_adjoint(dimage, k)
            for s, cell, gx, gy, x, y in self.taps(k):
                c = (h[cell].conj() * self.val[s]).real
                self.k.spread(out, x, c * gy)
                self.k.spread(out, y, c * gx)
        return out


def _exact_direct(case: dict, d: dict):
    u, v, w = (d[k].double() for k in ("u", "v", "w"))
    vis = torch.zeros(case["n_vis"], dtype=torch.complex128, device=DEV)

    def cis(ph):
        ph = (ph - ph.round()) * (2.0 * math.pi)
        return torch.complex(torch.cos(ph), torch.sin(ph))

    for l, m, f in zip(d["l"], d["m"], d["flux"]):
        vis += f * cis(-(u * l + v * m + w * (-(l * l + m * m) / (1.0 + math.sqrt(1.0 - l * l - m * m)))))
    val = vis if d["weight"] is None else vis * d["weight"].double()
    l = (d["pa"].double() - case["n"] // 2) * (case["fov"] / case["n"])
    m = (d["pb"].double() - case["n"] // 2) * (case["fov"] / case["n"])
    t = -(l * l + m * m) / (1.0 + torch.sqrt(1.0 - l * l - m * m))
    out = torch.zeros(case["pixels"], dtype=torch.complex128, device=DEV)
    step = max(1, (1 << 25) // case["pixels"])
    for a in range(0, case["n_vis"], step):
        s = slice(a, a + step)
        ph = torch.outer(l, u[s]) + torch.outer(m, v[s]) + torch.outer(t, w[s])
        out += cis(ph) @ val[s]
    return vis, out


def exact(case: dict, seed: int):
    d = _inputs(case, seed)
    if case["what"] == "direct":
        return _exact_direct(case, d)
    what, n = case["what"], case["n"]
    kernel = _Kernel(case)
    m = case["grid_n"] or n
    corr = 1.0 / kernel.transform(m)[(m - n) // 2:(m - n) // 2 + n]
    corr = corr[:, None] * corr[None, :]
    off = d["offsets"] or [0, case["n_vis"]]
    images = []
    for i in range(case["batch"]):
        s = slice(off[i], off[i + 1])
        geo = _Geometry(case, d["u"][s], d["v"][s], d["w"][s], d["vis"][s],
                        None if d["weight"] is None else d["weight"][s], kernel)
        if what == "degrid":
            return geo.degrid(d["dimage"][0].to(torch.complex128) * corr * geo.inside, case["n_vis"])
        img = geo.image()
        images.append(img if what == "table_grad" else img * corr)
    out = torch.stack(images)
    if what == "grad":
        return out, geo.degrid(d["dimage"][0].to(torch.complex128) * corr * geo.inside, case["n_vis"])
    if what == "table_grad":
        return out, geo.table_grad(d["dimage"][0].to(torch.complex128))
    return out
