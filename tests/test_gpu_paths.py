"""GPU behaviour and parity of branches that the other tests pass by.  Reference: the FP64
oracle; tolerances as in the other tests, 1e-5 of the largest value without grid correction
and 1e-4 for table gradients."""
import numpy as np
import pytest

import oracle
from oracle import OracleConfig
from paper_2301_06061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-5


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


def case(n, fov, n_vis, seed):
    rng = np.random.default_rng(seed)
    u, v, w = synth.disk_uvw(n_vis, 0.45 * n / fov, 150.0, rng)
    return u, v, w, synth.random_visibilities(n_vis, rng), rng


def configs(wst, n, fov, n_w, W=7, **kw):
    sigma = {7: 0.875, 8: 0.925}[W]
    return (wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kparam=sigma, **kw),
            OracleConfig(n, fov, n_w, -160.0, 160.0, W, "gauss", sigma))


@pytest.mark.parametrize("n", [64, 256, 2048])
@pytest.mark.parametrize("n_w,chunk", [(16, 0), (17, 0), (33, 0), (40, 0), (40, 20), (33, 7)])
def test_adjoint_over_many_planes(wst, n, n_w, chunk):
    """Degridding of one image where its planes make several runs of 16 (the screens' anchors
    are renewed, and runs go to blocks of their own where the tiles are few), whole and in
    chunks that cut runs."""
    fov = 0.1
    u, v, w, vis, rng = case(n, fov, 3000, [n, n_w, chunk])
    cfg, ocfg = configs(wst, n, fov, n_w, planes_per_chunk=chunk)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    y = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    got = plan.degrid(dev(y[None]), flags=wst.WST_NO_CORRECTION).cpu().numpy()
    want = oracle.degrid(ocfg, u, v, w, vis, y, correct=False)
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("chunk", [0, 20])
def test_adjoint_of_several_images_over_many_planes(wst, chunk):
    n, fov, n_w, batch, per = 256, 0.1, 18, 3, 1500
    u, v, w, vis, rng = case(n, fov, batch * per, chunk)
    cfg, ocfg = configs(wst, n, fov, n_w, batch=batch, planes_per_chunk=chunk)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), None, [per * i for i in range(batch + 1)])
    y = (rng.standard_normal((batch, n, n)) + 1j * rng.standard_normal((batch, n, n))).astype(np.complex64)
    got = plan.degrid(dev(y), flags=wst.WST_NO_CORRECTION).cpu().numpy()
    for i in range(batch):
        s = slice(per * i, per * (i + 1))
        want = oracle.degrid(ocfg, u[s], v[s], w[s], vis[s], y[i], correct=False)
        assert np.abs(got[s] - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("n,W,per_cell", [(512, 8, 511), (512, 8, 512), (512, 8, 1024), (256, 6, 512), (1024, 6, 1024),
                                          (512, 13, 512)])
def test_table_gradient_of_finely_sampled_tables(wst, n, W, per_cell):
    """From 512 samples per cell the first attempts of a record's additions go out together:
    half of the visibilities fall on a few positions, so that many lose the race and are added
    the usual way; supports with an instance of their own and taps in fours with a rest."""
    fov, n_w, n_vis = 0.1, 2, 4000
    u, v, w, vis, rng = case(n, fov, n_vis, [n, W, per_cell])
    h = n_vis // 2
    u[:h] = (rng.integers(0, 2, h) + 0.25).astype(np.float32) / np.float32(fov)
    v[:h] = np.float32(1.25 / fov)
    w[:h] = 10.0
    xs = np.linspace(-W / 2, W / 2, W * per_cell + 1)
    tab = (np.exp(-xs**2 / 1.7) * (1 + 0.05 * np.sin(xs))).astype(np.float32)
    plan = wst.Plan(wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kernel=wst.WST_KERNEL_TABLE,
                               ktable_len=tab.size))
    plan.set_kernel_table(dev(tab))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    ocfg = OracleConfig(n, fov, n_w, -160.0, 160.0, W, "table", 0.0, tab.astype(np.float64))
    y = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    got = plan.kernel_grad(dev(y[None])).cpu().numpy()
    ref = oracle.kernel_grad(ocfg, u, v, w, vis, y)
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("n", [64, 512, 1024, 4096, 16384])
def test_planes_between_alignments_are_refused(wst, n):
    """wst_fft_correct's passes copy 16 bytes at a time: planes that start 8 bytes past such a
    boundary are refused on the host, with the image untouched, and the plan stays usable."""
    u, v, w, vis, _ = case(n, 0.1, 10, n)
    plan = wst.Plan(configs(wst, n, 0.1, 1)[0])
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    raw = torch.zeros(n * n + 2, dtype=torch.complex64, device="cuda")
    img = torch.zeros((1, n, n), dtype=torch.complex64, device="cuda")
    with pytest.raises(wst.WstError) as e:
        wst.wst_fft_correct(plan.handle, 0, 1, raw[1:1 + n * n].view(1, n, n), img)
    assert wst.STATUS[e.value.status] == "WST_ERR_INVALID_ARG"
    assert not torch.view_as_real(img).any()
    wst.wst_fft_correct(plan.handle, 0, 1, raw[:n * n].view(1, n, n), img)
    assert not torch.view_as_real(img).any()


@pytest.mark.parametrize("n,batch,chunk", [(64, 7, 0), (512, 5, 4), (2048, 3, 4)])
def test_fp64_screens_of_several_images(wst, n, batch, chunk):
    fov, n_w, per = 0.1, 2, 1500
    u, v, w, vis, _ = case(n, fov, batch * per, [n, batch])
    cfg, ocfg = configs(wst, n, fov, n_w, batch=batch, planes_per_chunk=chunk, flags=wst.WST_FLAG_FP64_SCREEN)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), None, [per * i for i in range(batch + 1)])
    img = plan.image(flags=wst.WST_NO_CORRECTION).cpu().numpy()
    for i in range(batch):
        s = slice(per * i, per * (i + 1))
        ref = oracle.image(ocfg, u[s], v[s], w[s], vis[s], None, correct=False)
        assert np.abs(img[i] - ref).max() <= TOL * np.abs(ref).max()


def test_sort_clear_beyond_one_kernel(wst):
    """More than 4 MB of bucket counts are cleared by a memset (16385 planes' worth of 64 rows
    and up); bound twice, so that a count left over would show."""
    n, fov, n_w, batch = 64, 0.1, 4096, 5
    per = 4000
    u, v, w, vis, rng = case(n, fov, batch * per, 3)
    cfg, _ = configs(wst, n, fov, n_w, batch=batch, planes_per_chunk=64)
    plan = wst.Plan(cfg)
    off = [per * i for i in range(batch + 1)]
    for _ in range(2):
        w = rng.uniform(-150, 150, batch * per).astype(np.float32)
        plan.set_vis(dev(u), dev(v), dev(w), dev(vis), None, off)
        k = torch.empty(batch * per, dtype=torch.int32, device="cuda")
        i0, j0 = torch.empty_like(k), torch.empty_like(k)
        wst.wst_vis_cells(plan.handle, k, i0, j0)
        ko, io, jo, st = oracle.locate(OracleConfig(n, fov, n_w, -160.0, 160.0, 7, "gauss", 0.875), u, v, w, vis)
        np.testing.assert_array_equal(k.cpu().numpy(), ko)
        np.testing.assert_array_equal(i0.cpu().numpy(), io)
        np.testing.assert_array_equal(j0.cpu().numpy(), jo)
        assert plan.stats()["n_kept"] == int((st == 0).sum())


@pytest.mark.parametrize("n,W,grid_n", [(1024, 7, 0), (1024, 6, 0), (2048, 9, 0), (2048, 8, 0), (4096, 7, 0), (820, 6, 1024),
                                        (1640, 8, 2048)])
@pytest.mark.parametrize("ratio", [95.0, 105.0])
def test_images_at_both_sides_of_the_integer_rule(wst, n, W, grid_n, ratio):
    """Rows of 1024 to 4096 are summed in integers where the grid correction raises an image's
    edge by less than 100, else in float (supports without an instance of their own then by
    rows in step): a Gaussian exp(-x^2 / 2 sigma^2) raises it by exp((pi sigma n / M)^2 / 2).
    The bins of the integer path show in the workspace."""
    fov, n_vis, n_w = 0.1, 9000, 2
    m = grid_n or n
    sigma = np.sqrt(2.0 * np.log(ratio)) / np.pi * m / n
    u, v, w, vis, rng = case(n, fov, n_vis, [n, W, int(ratio)])
    cfg = wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=16, kparam=sigma, grid_n=grid_n)
    bins = 4 * n_w * m * m // 64
    size = wst.wst_plan_workspace_bytes(wst.Plan(cfg).handle, n_vis)
    other = wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=16, kparam=2 * sigma, grid_n=grid_n)
    float_size = wst.wst_plan_workspace_bytes(wst.Plan(other).handle, n_vis)
    assert (size >= float_size + bins) if ratio < 100 else size == float_size
    # the narrower kernel's image (its edge is cut off at W/2, which leaves the side it is on)
    cfg.support = W
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    img = plan.image(flags=wst.WST_NO_CORRECTION)[0].cpu().numpy()
    ocfg = OracleConfig(n, fov, n_w, -160.0, 160.0, W, "gauss", sigma)
    ref = oracle.image_on_grid(ocfg, m, u, v, w, vis, None, correct=False)
    assert np.abs(img - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("n", [64, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("W,chunk", [(5, 0), (8, 2), (16, 1)])
def test_planes_of_every_row_length(wst, n, W, chunk):
    """wst_grid, whose rows of 512 to 2048 are worked on in step: empty rows, rows at the mesh's
    edges, plane ranges that do not start at the first plane."""
    fov, n_w = 0.1, 3
    u, v, w, vis, rng = case(n, fov, 4000, [n, W])
    v[:2000] *= 0.01  # most rows empty, a few busy
    v[-50:] = np.float32((0.5 * n - 0.5 * W - 0.01) / fov)
    wt = rng.uniform(0.25, 2.0, 4000).astype(np.float32)
    sigma = 0.875 * np.sqrt(W / 7.0)
    plan = wst.Plan(wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kparam=sigma))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), dev(wt))
    ref = oracle.grid(OracleConfig(n, fov, n_w, -160.0, 160.0, W, "gauss", sigma), u, v, w, vis, wt)
    g = torch.full((n_w, n, n), float("nan"), dtype=torch.complex64, device="cuda")
    for a, b in [(0, n_w)] if not chunk else [(k, min(k + chunk, n_w)) for k in range(0, n_w, chunk)]:
        wst.wst_grid(plan.handle, a, b, g[a:b])
    assert np.abs(g.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("n", [64, 128, 256, 512])
@pytest.mark.parametrize("W", [7, 9])
@pytest.mark.parametrize("more", [-1, 0])
def test_short_rows_below_and_from_two_rounds_of_blocks(wst, n, W, more):
    """Float rows shorter than 1024 are worked on in step from two rounds of blocks (four of
    4096 / N rows per SM) on, by groups below: images and planes at both sides, some planes and
    rows without visibilities."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_w, fov = 2 * 4 * sms * 4096 // (n * n) + more, 0.1
    u, v, w, vis, rng = case(n, fov, 6000, [n, W])
    v[:3000] *= 0.01
    w[:1000] = 3.0
    wt = rng.uniform(0.25, 2.0, 6000).astype(np.float32)
    sigma = 0.875 * np.sqrt(W / 7.0)
    plan = wst.Plan(wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kparam=sigma))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), dev(wt))
    ocfg = OracleConfig(n, fov, n_w, -160.0, 160.0, W, "gauss", sigma)
    img = plan.image(flags=wst.WST_NO_CORRECTION)[0].cpu().numpy()
    ref = oracle.image(ocfg, u, v, w, vis, wt, correct=False)
    assert np.abs(img - ref).max() <= TOL * np.abs(ref).max()
    g = torch.full((n_w, n, n), float("nan"), dtype=torch.complex64, device="cuda")
    wst.wst_grid(plan.handle, 0, n_w, g)
    ref = oracle.grid(ocfg, u, v, w, vis, wt)
    assert np.abs(g.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("n", [1024, 2048, 4096])
def test_rows_too_dense_for_the_integer_bound(wst, n):
    """Rows whose busiest 64 columns hold more than 8192 times the row's mean magnitude go
    straight to float sums, beside ordinary rows in integers (300,000 values over three bins
    of seven rows)."""
    fov, dense, rest = 0.1, 300_000, 20_000
    rng = np.random.default_rng(n)
    u = (np.concatenate([rng.uniform(-90.0, 90.0, dense), rng.uniform(-0.45, 0.45, rest) * n]) / fov).astype(np.float32)
    v = (np.concatenate([np.zeros(dense), rng.uniform(-0.45, 0.45, rest) * n]) / fov).astype(np.float32)
    w = rng.uniform(-10.0, 10.0, dense + rest).astype(np.float32)
    vis = synth.random_visibilities(dense + rest, rng)
    plan = wst.Plan(wst.Config(n=n, fov=fov, n_w=1, w_min=-10.0, w_max=10.0))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    img = plan.image(flags=wst.WST_NO_CORRECTION)[0].cpu().numpy()
    ref = oracle.image(OracleConfig(n, fov, 1, -10.0, 10.0, 7, "gauss", 0.875), u, v, w, vis, None, correct=False)
    assert np.abs(img - ref).max() <= TOL * np.abs(ref).max()
