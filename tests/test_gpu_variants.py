"""GPU parity of single kernels at the sizes where their code takes another turn: edges of
blocks and tiles, remainders, the smallest and largest of a range.  References: the FP64
oracle, or the same formula in numpy FP64."""
import numpy as np
import pytest

import oracle
from oracle import OracleConfig
from paper_2301_06061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wst():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_06061_gb300 import build, wst as w

    build.build()
    w.load_library()
    return w


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ------------------------------------------------------------------------------------------
# grid correction 1/Ghat
# ------------------------------------------------------------------------------------------

def simpson_ghat(g_ends, g_mid, W, n):
    """Composite Simpson of G(x) cos(2 pi nu x) over panels with the kernel's values at the
    panel ends (P + 1) and middles (P); also the sum of the weights' magnitudes."""
    P = len(g_mid)
    x = np.linspace(-0.5 * W, 0.5 * W, 2 * P + 1)
    g = np.empty(2 * P + 1)
    g[::2], g[1::2] = g_ends, g_mid
    wt = np.full(2 * P + 1, 2.0)
    wt[1::2] = 4.0
    wt[0] = wt[-1] = 1.0
    c = wt * g * (W / P / 6.0)
    nu = (np.arange(n) - n // 2) / n
    return np.cos(2.0 * np.pi * np.outer(nu, x)) @ c, np.abs(c).sum()


@pytest.mark.parametrize("n", [64, 1024])
@pytest.mark.parametrize("kernel,W,length", [("gauss", 7, 0), ("es", 2, 0), ("table", 2, 2), ("table", 3, 128),
                                             ("table", 8, 129), ("table", 8, 8193)])
def test_correction_is_composite_simpson(wst, n, kernel, W, length):
    """Every 1/Ghat is the FP64 quadrature rounded to FP32 (also for tables that are not
    symmetric).  wst_correct of a unit image gives corr_a corr_b; along the central row the
    products carry three FP32 roundings, 3 * 2^-24; the FP64 sum's own error is taken as
    1e-12 of the sum of the weights."""
    half = 0.5 * W
    if kernel == "table":
        rng = np.random.default_rng(length)
        tab = (1.0 + rng.random(length)).astype(np.float32)
        cfg = wst.Config(n=n, fov=0.1, n_w=1, support=W, kernel=wst.WST_KERNEL_TABLE, ktable_len=length)
        t = tab.astype(np.float64)
        want, total = simpson_ghat(t, 0.5 * (t[1:] + t[:-1]), W, n)
    else:
        P = 256 * W
        x = np.linspace(-half, half, 2 * P + 1)
        par = 0.875 if kernel == "gauss" else 2.3 * W
        g = np.exp(-x * x / (2 * par * par)) if kernel == "gauss" else \
            np.exp(par * (np.sqrt(np.clip(1 - (x / half) ** 2, 0, None)) - 1))
        cfg = wst.Config(n=n, fov=0.1, n_w=1, support=W, kernel=0 if kernel == "gauss" else 1, kparam=par)
        want, total = simpson_ghat(g[::2], g[1::2], W, n)
    plan = wst.Plan(cfg)
    if kernel == "table":
        plan.set_kernel_table(dev(tab))
    img = torch.ones((1, n, n), dtype=torch.complex64, device="cuda")
    wst.wst_plan_stream(plan.handle)
    wst.wst_correct(plan.handle, img)
    prod = img[0, n // 2].real.double().cpu().numpy()  # corr_{n/2} corr_a
    got = 1.0 / (prod * want[n // 2])
    assert np.all(np.abs(got - want) <= 3 * 2.0 ** -24 * np.abs(want) * 1.01 + 1e-12 * total)


# ------------------------------------------------------------------------------------------
# sort: visibilities of uneven images over the blocks
# ------------------------------------------------------------------------------------------

@pytest.mark.parametrize("counts", [[1], [31, 0, 33], [0, 1, 31, 33, 0, 5000, 2, 0, 70_000, 64], [1] * 130])
def test_sort_of_uneven_images(wst, counts):
    """Placement, counts and each image's w range (from the data) against the oracle, where
    a block's share of the visibilities spans several images, empty ones among them."""
    n, fov, n_w = 256, 0.1, 5
    total = sum(counts)
    u, v, w = synth.disk_uvw(total, 0.53 * n / fov, 150.0, np.random.default_rng(total))
    vis = synth.random_visibilities(total, np.random.default_rng(1))
    vis[::97] = np.nan
    off = [0] + [int(x) for x in np.cumsum(counts)]
    plan = wst.Plan(wst.Config(n=n, fov=fov, n_w=n_w, batch=len(counts)))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), None, off)
    k = torch.empty(total, dtype=torch.int32, device="cuda")
    i0, j0 = torch.empty_like(k), torch.empty_like(k)
    wst.wst_vis_cells(plan.handle, k, i0, j0)
    kept = dropped = bad = 0
    for a, b in zip(off[:-1], off[1:]):
        lo, hi = oracle.resolve_w_range(w[a:b], 0.0, 0.0)
        ko, io, jo, st = oracle.locate(OracleConfig(n, fov, n_w, lo, hi), u[a:b], v[a:b], w[a:b], vis[a:b])
        np.testing.assert_array_equal(k[a:b].cpu().numpy(), ko)
        np.testing.assert_array_equal(i0[a:b].cpu().numpy(), io)
        np.testing.assert_array_equal(j0[a:b].cpu().numpy(), jo)
        kept, dropped, bad = kept + int((st == 0).sum()), dropped + int((st == 1).sum()), bad + int((st == 2).sum())
    s = plan.stats()
    assert (s["n_kept"], s["n_dropped"], s["n_nonfinite"]) == (kept, dropped, bad)


# ------------------------------------------------------------------------------------------
# direct transforms
# ------------------------------------------------------------------------------------------

@pytest.mark.parametrize("n_vis,n_pix", [(1, 1), (255, 8), (257, 9), (3001, 17), (40_000, 7)])
def test_direct_transforms_against_fp64(wst, n_vis, n_pix):
    """wst_dft and wst_predict_points on a field reaching outside the unit sphere, with (u, v,
    w) from below one to thousands of cycles of phase.  Per visibility the phase is rounded
    to FP32 twice at magnitude <= 1 (2^-24 cycle each) and sincospi errs by 2^-22 at most; a
    thread adds n_vis/256 terms and the reduction 20 more, each rounding by 2^-24 of a
    partial sum; the output's magnitude bound is sum |w V|."""
    n, fov = 4096, 1.9
    rng = np.random.default_rng(n_vis)
    scale = 10.0 ** rng.uniform(-2, 3.5, (3, n_vis))
    u, v, w = (scale * rng.uniform(-1, 1, (3, n_vis))).astype(np.float32)
    vis = synth.random_visibilities(n_vis, rng)
    wt = rng.uniform(0.5, 1.5, n_vis).astype(np.float32)
    pa, pb = rng.integers(0, n, (2, n_pix)).astype(np.int32)
    pa[0], pb[0] = n // 2, n // 2  # the phase centre
    if n_pix > 1:
        pa[1], pb[1] = 0, 0  # outside the unit sphere
    out = torch.full((n_pix,), float("nan"), dtype=torch.complex64, device="cuda")
    wst.wst_dft(dev(u), dev(v), dev(w), dev(vis), n, fov, dev(pa), dev(pb), out, dev(wt))
    ref = oracle.dft_pixels(u, v, w, vis, n, fov, pa, pb, wt)
    per_vis = 2 * np.pi * 2 * 2.0 ** -24 + 2.0 ** -22
    tol = (per_vis + 2.0 ** -24 * (n_vis / 256 + 21)) * np.abs(wt * vis).sum()
    assert np.abs(out.cpu().numpy() - ref).max() <= tol
    if n_pix > 1:
        assert out[1] == 0
    l, m = rng.uniform(-0.6, 0.6, (2, n_pix))
    flux = rng.uniform(0.1, 1.0, n_pix)
    got = torch.empty(n_vis, dtype=torch.complex64, device="cuda")
    wst.wst_predict_points(dev(u), dev(v), dev(w), dev(l), dev(m), dev(flux), got)
    err = np.abs(got.cpu().numpy() - oracle.predict_points(u, v, w, l, m, flux)).max()
    assert err <= (per_vis + 2.0 ** -24 * (n_pix + 1)) * flux.sum()


@pytest.mark.parametrize("scale", [0.99, 1.01, 4.0])
def test_direct_transforms_around_the_fast_phases_range(wst, scale):
    """|u| at and beyond 2^20 wavelengths, where the direct transforms change to the general
    phase reduction, with sources in and outside |l| <= 1 for the prediction.  l is a pair of
    floats, 2^-49 of its value, so a phase errs by 2^-29 cycle there; the sums' bound is that
    of the phases' FP32 rounding."""
    n, fov, n_vis, n_pix = 512, 0.2, 3000, 9
    rng = np.random.default_rng(int(100 * scale))
    u, v, w = (rng.uniform(-1, 1, (3, n_vis)) * scale * 2.0 ** 20).astype(np.float32)
    vis = synth.random_visibilities(n_vis, rng)
    pa, pb = rng.integers(0, n, (2, n_pix)).astype(np.int32)
    out = torch.empty(n_pix, dtype=torch.complex64, device="cuda")
    wst.wst_dft(dev(u), dev(v), dev(w), dev(vis), n, fov, dev(pa), dev(pb), out)
    ref = oracle.dft_pixels(u, v, w, vis, n, fov, pa, pb)
    per_vis = 2 * np.pi * 3 * 2.0 ** -24 + 2.0 ** -22
    assert np.abs(out.cpu().numpy() - ref).max() <= (per_vis + 2.0 ** -24 * (n_vis / 256 + 21)) * np.abs(vis).sum()
    for far in (0.0, 1.5):
        l, m = rng.uniform(-0.1, 0.1, (2, 5))
        l[0] += far
        flux = rng.uniform(0.1, 1.0, 5)
        got = torch.empty(n_vis, dtype=torch.complex64, device="cuda")
        wst.wst_predict_points(dev(u), dev(v), dev(w), dev(l), dev(m), dev(flux), got)
        keep = np.arange(5) if far == 0.0 else np.arange(1, 5)
        if far == 0.0:
            err = np.abs(got.cpu().numpy() - oracle.predict_points(u, v, w, l, m, flux)).max()
            assert err <= (per_vis + 2.0 ** -24 * 6) * flux[keep].sum()
        else:
            assert torch.isfinite(torch.view_as_real(got)).all()
