"""GPU results held to FP32 precision where a shared quantum, a summation order or a reduced
argument could take bits from them.  References: the FP64 oracle, or the same formula in
numpy FP64; each test derives its bound."""
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
# gridder
# ------------------------------------------------------------------------------------------

def assert_cells(wst, cfg, ocfg, u, v, w, vis, adds, rows=slice(None)):
    """Every cell of the given rows of wst_grid's planes within FP32 of its own terms: |error| <= eps S with S the
    sum of the terms' magnitudes in that cell, eps = (adds + 32) 2^-24 (`adds` roundings of
    partial sums; 32 for the two taps, whose argument of up to 4 cells is rounded to 2^-24
    cell under a slope of at most 5 per cell, their exponentials and the products)."""
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    g = torch.empty((cfg.n_w, cfg.n, cfg.n), dtype=torch.complex64, device="cuda")
    wst.wst_grid(plan.handle, 0, cfg.n_w, g)
    got = g.cpu().numpy()[:, rows]
    ref = oracle.grid(ocfg, u, v, w, vis)[:, rows]
    size = oracle.grid(ocfg, u, v, w, (np.abs(vis.real) + np.abs(vis.imag)).astype(np.complex64))[:, rows].real
    assert np.all(np.abs(got - ref) <= (adds + 32) * 2.0 ** -24 * size)


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("W", [6, 7, 8])
def test_cells_far_below_a_bright_one(wst, n, W):
    """300 values of order one and one of 1e6 in the same rows: the other cells keep their own
    precision (a quantum taken from the rows' brightest bin would leave them ten bits)."""
    rng = np.random.default_rng([n, W])
    fov, n_vis = 0.1, 301
    u = (rng.uniform(-0.4, 0.4, n_vis) * n / fov).astype(np.float32)
    v = np.full(n_vis, 3.3 / fov, np.float32)
    w = np.zeros(n_vis, np.float32)
    vis = synth.random_visibilities(n_vis, rng)
    vis[0] = 1e6
    sigma = {6: 0.81, 7: 0.875, 8: 0.925}[W]
    cfg = wst.Config(n=n, fov=fov, n_w=1, w_min=-10.0, w_max=10.0, support=W, kparam=sigma)
    ocfg = OracleConfig(n, fov, 1, -10.0, 10.0, W, "gauss", sigma)
    assert_cells(wst, cfg, ocfg, u, v, w, vis, adds=301 if n == 64 else 64)


@pytest.mark.parametrize("n", [64, 256, 2048, 8192])
@pytest.mark.parametrize("W", [6, 8])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_kernel_samples_show(wst, n, W, bad):
    """A kernel table that has diverged shows in the gridded planes and the uncorrected image:
    integer sums must not swallow it."""
    per_cell = 4
    rng = np.random.default_rng(n + W)
    u, v, w = synth.disk_uvw(500, 0.3 * n / 0.1, 5.0, rng)
    tab = np.ones(W * per_cell + 1, np.float32)
    tab[W * per_cell // 2 - 1] = bad
    plan = wst.Plan(wst.Config(n=n, fov=0.1, n_w=1, w_min=-10.0, w_max=10.0, support=W, kernel=wst.WST_KERNEL_TABLE,
                               ktable_len=tab.size))
    plan.set_kernel_table(dev(tab))
    plan.set_vis(dev(u), dev(v), dev(w), dev(synth.random_visibilities(500, rng)))
    g = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
    wst.wst_grid(plan.handle, 0, 1, g)
    assert not torch.isfinite(torch.view_as_real(g)).all()
    assert not torch.isfinite(torch.view_as_real(plan.image(flags=wst.WST_NO_CORRECTION))).all()


@pytest.mark.parametrize("W", [7, 8])
def test_faint_cells_of_a_row_that_leaves_the_integer_range(wst, W):
    """Rows of 8192 whose coherent pile-up of 400 equal values on one cell wraps the integer
    sums, with 400 values of 1e-4 over the rest of them: summed again in float, the faint cells
    keep their own precision.  The range holds an eighth of a bin's magnitude, 50; with a tap
    G_x = 0.96 for the pile-up the rows with G_y >= 0.15 pass it."""
    rng = np.random.default_rng(W)
    n, fov, k = 8192, 0.1, 400
    u = np.concatenate([np.full(k, 300.25), rng.uniform(-0.4, 0.4, k) * n]).astype(np.float32) / np.float32(fov)
    v = np.full(2 * k, 3.3 / fov, np.float32)
    w = np.zeros(2 * k, np.float32)
    vis = np.concatenate([np.full(k, 1.0 + 0.5j), 1e-4 * synth.random_visibilities(k, rng)]).astype(np.complex64)
    sigma = {7: 0.875, 8: 0.925}[W]
    cfg = wst.Config(n=n, fov=fov, n_w=1, w_min=-10.0, w_max=10.0, support=W, kparam=sigma)
    y = np.arange(n) - (n // 2 + 3.3)
    rows = np.flatnonzero(np.exp(-y * y / (2 * sigma * sigma)) >= 0.15)
    assert len(rows) >= 3
    assert_cells(wst, cfg, OracleConfig(n, fov, 1, -10.0, 10.0, W, "gauss", sigma), u, v, w, vis, adds=400, rows=rows)


# ------------------------------------------------------------------------------------------
# degridding
# ------------------------------------------------------------------------------------------

@pytest.mark.parametrize("n,n_vis", [(512, 60_000), (2048, 30_000), (2048, 1_000_000), (4096, 2_000_000),
                                     (8192, 3_000_000)])
def test_row_sums_added_in_order(wst, n, n_vis):
    """The W row sums of a visibility added from its first tap row to its last.  The image is
    one pixel on the field's edge and the kernel is flat, so the row sums are exactly +c, -c,
    +c, ... with c = fl(W weight): in order (or with neighbours exchanged) every partial sum
    is a multiple of c up to 2c, exact, and the result is +-c to the last bit.  Orders at random
    round the sums of one in eight (simulated below); a tenth of that is left to rows that
    overtake each other."""
    fov, W = 0.1, 7
    rng = np.random.default_rng(n)
    u, v, _ = synth.disk_uvw(n_vis, 0.45 * n / fov, 150.0, rng)
    wt = rng.uniform(0.5, 1.5, n_vis).astype(np.float32)
    cfg = wst.Config(n=n, fov=fov, n_w=1, w_min=-10.0, w_max=10.0, support=W, kernel=wst.WST_KERNEL_TABLE,
                     ktable_len=W + 1)
    plan = wst.Plan(cfg)
    plan.set_kernel_table(torch.ones(W + 1, device="cuda"))
    plan.set_vis(dev(u), dev(v), dev(np.zeros_like(u)), dev(np.ones(n_vis, np.complex64)), dev(wt))
    y = torch.zeros((1, n, n), dtype=torch.complex64, device="cuda")
    y[0, 0, n // 2] = 1.0
    got = plan.degrid(y, flags=wst.WST_NO_CORRECTION).cpu().numpy()
    c = np.float32(W) * wt
    assert not got.imag.any() and np.abs(np.abs(got.real) - c).max() <= W * 2.0 ** -22 * c.max()
    some = c[:20_000]
    signs = rng.permuted(np.tile(np.array([1, -1, 1, -1, 1, -1, 1], np.float32), (len(some), 1)), axis=1)
    acc = np.zeros_like(some)
    for k in range(W):
        acc += signs[:, k] * some
    assert np.mean(np.abs(got.real) != c) <= 0.1 * np.mean(acc != some)


# ------------------------------------------------------------------------------------------
# direct transforms
# ------------------------------------------------------------------------------------------

def test_sine_and_cosine(wst):
    """The direct transforms' (and the screens') sine and cosine alone: one source at l = 1/2
    makes the phase u / 2, exact in FP32.  The evaluation errs by less than 2^-24, the spacing
    of the results just below one."""
    u = np.linspace(-1.5, 1.5, 3_000_001).astype(np.float32)
    zero = dev(np.zeros_like(u))
    got = torch.empty(u.size, dtype=torch.complex64, device="cuda")
    one = dev(np.ones(1))
    wst.wst_predict_points(dev(u), zero, zero, 0.5 * one, 0.0 * one, one, got)
    got = got.cpu().numpy()
    phase = -np.pi * u.astype(np.float64)
    assert np.abs(got.real - np.cos(phase)).max() < 2.0 ** -24
    assert np.abs(got.imag - np.sin(phase)).max() < 2.0 ** -24


@pytest.mark.parametrize("scale", [100.0, 2.0 ** 14, 2.0 ** 17, 1.01 * 2.0 ** 19, 2.0 ** 20])
@pytest.mark.parametrize("far", [False, True])
def test_phases_in_float_float(wst, scale, far):
    """The phase u l + v m + w (n - 1) in float-float, at and beyond the range that takes it
    without renormalisations, and from a source outside the unit sphere (n - 1 counts as
    zero there).  It is rounded to FP32 once, below or just above half a cycle: 2^-25 cycle;
    l, m and n - 1 are pairs of floats, 2^-48 of a coordinate; the sine and cosine err by
    2^-24 at most."""
    rng = np.random.default_rng(int(scale) + far)
    n_vis = 400_000
    u, v, w = rng.uniform(-scale, scale, (3, n_vis)).astype(np.float32)
    for _ in range(3):
        l, m = rng.uniform(-0.6, 0.6, 2)
        if far:
            l += 1.5
        r2 = l * l + m * m
        t = -r2 / (1.0 + np.sqrt(1.0 - r2)) if r2 < 1.0 else 0.0
        got = torch.empty(n_vis, dtype=torch.complex64, device="cuda")
        wst.wst_predict_points(dev(u), dev(v), dev(w), dev(np.array([l])), dev(np.array([m])), dev(np.ones(1)), got)
        phase = u.astype(np.longdouble) * l + v.astype(np.longdouble) * m + w.astype(np.longdouble) * t
        phase = (phase - np.rint(phase)).astype(np.float64) * (-2.0 * np.pi)
        err = got.cpu().numpy() - np.exp(1j * phase)
        tol = 2.0 * np.pi * (2.0 ** -25 + 3.0 * scale * 2.0 ** -48) + 2.0 ** -24
        assert max(np.abs(err.real).max(), np.abs(err.imag).max()) <= tol


def test_direct_transform_phases(wst):
    """The same for wst_dft at single visibilities: one visibility, every pixel its phase."""
    n, fov, n_pix = 4096, 0.9, 4096
    rng = np.random.default_rng(5)
    pa, pb = rng.integers(0, n, (2, n_pix)).astype(np.int32)
    l, m = (pa - n // 2) * (fov / n), (pb - n // 2) * (fov / n)
    t = -(l * l + m * m) / (1.0 + np.sqrt(1.0 - l * l - m * m))
    for scale in [3e3, 1e5]:
        u, v, w = rng.uniform(-scale, scale, (3, 1)).astype(np.float32)
        out = torch.empty(n_pix, dtype=torch.complex64, device="cuda")
        wst.wst_dft(dev(u), dev(v), dev(w), dev(np.ones(1, np.complex64)), n, fov, dev(pa), dev(pb), out)
        phase = u.astype(np.longdouble) * l + v.astype(np.longdouble) * m + w.astype(np.longdouble) * t
        phase = (phase - np.rint(phase)).astype(np.float64) * (2.0 * np.pi)
        err = out.cpu().numpy() - np.exp(1j * phase)
        tol = 2.0 * np.pi * (2.0 ** -25 + 3.0 * scale * 2.0 ** -48) + 2.0 ** -24
        assert max(np.abs(err.real).max(), np.abs(err.imag).max()) <= tol


# ------------------------------------------------------------------------------------------
# grid correction
# ------------------------------------------------------------------------------------------

@pytest.mark.parametrize("W,per_cell", [(16, 4095), (16, 2048), (8, 1024), (10, 128)])
def test_correction_where_the_transform_is_small(wst, W, per_cell):
    """1/Ghat of unpadded Kaiser-Bessel tables, whose transform falls to 1e-6 ... 1e-10 of
    Ghat(0) at the field's edge.  wst_correct of a unit image gives corr_a corr_b: three FP32
    roundings along the central row.  Beside them Ghat may err by the roundings of an FP64 sum:
    each is 2^-53 of a partial sum, and over a thousand terms and more they average out to
    an eighth of 2^-53 of the terms' magnitudes or less."""
    from paper_2301_06061_gb300 import kernels

    n, length = 64, W * per_cell + 1
    tab = kernels.kaiser_bessel_table(W, kernels.kaiser_bessel_beta(W), per_cell)
    assert len(tab) == length
    t = tab.astype(np.float64)
    x = np.linspace(-0.5 * W, 0.5 * W, 2 * length - 1)
    g = np.empty(2 * length - 1)
    g[::2], g[1::2] = t, 0.5 * (t[1:] + t[:-1])
    wt = np.full(g.size, 2.0)
    wt[1::2] = 4.0
    wt[0] = wt[-1] = 1.0
    c = wt * g * (1.0 / per_cell / 6.0)
    at = np.array([0, 1, 2, 3, 4, 8, 16, 31, 32])
    pi = np.longdouble("3.14159265358979323846264338327950288")
    want = np.array([np.sum(np.cos(2 * pi * (a - n // 2) / n * x.astype(np.longdouble)) * c) for a in at])
    want = want.astype(np.float64)
    plan = wst.Plan(wst.Config(n=n, fov=0.1, n_w=1, support=W, kernel=wst.WST_KERNEL_TABLE, ktable_len=length))
    plan.set_kernel_table(dev(tab))
    img = torch.ones((1, n, n), dtype=torch.complex64, device="cuda")
    wst.wst_plan_stream(plan.handle)
    wst.wst_correct(plan.handle, img)
    prod = img[0, n // 2, at].real.double().cpu().numpy()
    got = 1.0 / (prod * want[-1])
    assert np.all(np.abs(got - want) <= 3 * 2.0 ** -24 * np.abs(want) * 1.01 + 2.0 ** -56 * np.abs(c).sum())


# ------------------------------------------------------------------------------------------
# workspace
# ------------------------------------------------------------------------------------------

@pytest.mark.parametrize("flags", [0, "fold"])
@pytest.mark.parametrize("n", [256, 2048])
def test_workspace_per_visibility(wst, n, flags):
    """Below the planes' size only the sorted records (32 bytes) grow with the visibilities, at
    any count: no second array of sums, least of all in a plan that cannot degrid."""
    cfg = wst.Config(n=n, fov=0.1, n_w=2048 // n * 16, flags=wst.WST_FLAG_WFOLD if flags else 0)
    plan = wst.Plan(cfg)
    size = [wst.wst_plan_workspace_bytes(plan.handle, k) for k in (1000, 200_000, 600_000)]
    planes = 8 * cfg.n_w * n * n
    assert 32 * 600_000 <= planes  # the sort's keys fit the planes' place
    assert size[1] - size[0] <= 32 * 199_000 + 256
    assert size[2] - size[0] <= 32 * 599_000 + 256


def test_table_gradient_takes_what_a_row_leaves(wst):
    """At 16384 a table of 6972 samples fits the row kernel's shared memory beside the row and
    its twiddles.  A flat table and one visibility at the phase centre, of value one: tap
    (a, d) contributes Re(conj(gh) V) = 1 (the image is one pixel at the centre, its transform
    one everywhere) to both its profiles, W of them each; every tap's share goes to the two
    samples around it, so W^2 lands on the x profile and W^2 on the y profile."""
    n, W, length = 16384, 7, 6972
    plan = wst.Plan(wst.Config(n=n, fov=0.1, n_w=1, w_min=-10.0, w_max=10.0, support=W, kernel=wst.WST_KERNEL_TABLE,
                               ktable_len=length))
    plan.set_kernel_table(torch.ones(length, device="cuda"))
    zero = torch.zeros(1, device="cuda")
    plan.set_vis(zero, zero, zero, torch.ones(1, dtype=torch.complex64, device="cuda"))
    y = torch.zeros((1, n, n), dtype=torch.complex64, device="cuda")
    y[0, n // 2, n // 2] = 1.0
    grad = plan.kernel_grad(y)
    assert abs(float(grad.double().sum()) - 2 * W * W) < 1e-4
