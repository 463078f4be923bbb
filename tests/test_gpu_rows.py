"""GPU parity of the row kernels (gridding and its adjoint fused with the row FFT) and of the
column passes at every line length, around the group, batch and quantum decisions they take.
Reference: the FP64 oracle.  Tolerance: 1e-5 of the largest value without grid correction,
the accuracy stated for FP32 results throughout; table gradients 1e-4, as elsewhere."""
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


def coords(kind: str, n: int, fov: float, n_vis: int, rng):
    """'disk': over most of the mesh and past its edges.  'cluster': half of the visibilities
    on a few cells, equal and in phase (partial sums leave the fine quantum's range), the
    rest spread.  'single': one visibility.  'edge': tap starts on the mesh's first and last
    rows and columns."""
    u, v, w = synth.disk_uvw(n_vis, 0.52 * n / fov, 150.0, rng)
    vis = synth.random_visibilities(n_vis, rng)
    if kind == "cluster":
        h = n_vis // 2
        u[:h] = (rng.integers(0, 2, h) + 0.25).astype(np.float32) / np.float32(fov)
        v[:h] = np.float32(1.25 / fov)
        w[:h] = 10.0
        vis[:h] = 1.0 + 0.5j
    elif kind == "edge":
        side = np.float32((0.5 * n - 4.01) / fov)
        u = np.where(rng.random(n_vis) < 0.5, -side, side).astype(np.float32)
        v = np.where(rng.random(n_vis) < 0.5, -side, side).astype(np.float32)
    return u, v, w, vis


def config(wst, n, fov, n_w, W, kernel="gauss", **kw):
    sigma = {7: 0.875, 8: 0.925}.get(W, 0.875 * (W / 7.0) ** 0.5)
    par = sigma if kernel == "gauss" else 2.3 * W
    kind = wst.WST_KERNEL_GAUSS if kernel == "gauss" else wst.WST_KERNEL_ES
    return (wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kernel=kind, kparam=par, **kw),
            OracleConfig(n, fov, n_w, -160.0, 160.0, W, kernel, par))


@pytest.mark.parametrize("kind,n_vis", [("disk", 9000), ("cluster", 9000), ("single", 1), ("edge", 300)])
@pytest.mark.parametrize("n,W,kernel", [(64, 7, "gauss"), (128, 5, "gauss"), (256, 8, "gauss"), (512, 7, "gauss"),
                                        (512, 6, "es"), (1024, 8, "es"), (1024, 16, "gauss"), (2048, 7, "gauss"),
                                        (4096, 8, "gauss"), (4096, 2, "gauss")])
def test_image_and_adjoint_at_every_row_length(wst, n, W, kernel, kind, n_vis):
    fov, n_w = 0.1, 3
    rng = np.random.default_rng([n, W, n_vis])
    u, v, w, vis = coords(kind, n, fov, n_vis, rng)
    wt = rng.uniform(0.25, 2.0, n_vis).astype(np.float32)
    cfg, ocfg = config(wst, n, fov, n_w, W, kernel, planes_per_chunk=2)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), dev(wt))
    ref = oracle.image(ocfg, u, v, w, vis, wt, correct=False)
    img = plan.image(flags=wst.WST_NO_CORRECTION)[0].cpu().numpy()
    assert np.abs(img - ref).max() <= TOL * np.abs(ref).max()
    y = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    got = plan.degrid(dev(y[None]), flags=wst.WST_NO_CORRECTION).cpu().numpy()
    want = oracle.degrid(ocfg, u, v, w, vis, y, wt, correct=False)
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("n_vis", [(1 << 19) - 1, 1 << 19])
def test_degrid_in_either_summing_order(wst, n_vis):
    """At the count from which the sums are kept in sorted order, and one below it; dropped and
    non-finite visibilities get zeros."""
    n, fov, n_w, W = 512, 0.1, 2, 7
    rng = np.random.default_rng(n_vis)
    u, v, w = synth.disk_uvw(n_vis, 0.53 * n / fov, 150.0, rng)
    vis = synth.random_visibilities(n_vis, rng)
    vis[::1001] = np.nan
    cfg, ocfg = config(wst, n, fov, n_w, W)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    y = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    want = oracle.degrid(ocfg, u, v, w, vis, y, correct=False)
    for _ in range(2):
        got = plan.degrid(dev(y[None]), flags=wst.WST_NO_CORRECTION).cpu().numpy()
        assert np.abs(got - want).max() <= TOL * np.abs(want).max()
        assert not got[::1001].any()
    # an output that starts between two complex numbers' alignments (C callers)
    raw = torch.empty(2 * n_vis + 1, dtype=torch.float32, device="cuda")
    from paper_2301_06061_gb300.wst import WST_NO_CORRECTION, load_library
    st = load_library().wst_degrid(plan.handle, dev(y[None]).data_ptr(), raw.data_ptr() + 4, WST_NO_CORRECTION)
    odd = torch.view_as_complex(raw[1:].clone().view(-1, 2)).cpu().numpy()
    assert st == 0 and np.abs(odd - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("n,batch,chunk,crop", [(64, 7, 0, 0), (256, 5, 4, 0), (512, 9, 0, 0), (512, 4, 3, 410),
                                                (2048, 3, 0, 0), (2048, 2, 3, 1640)])
def test_images_of_one_call_split_over_blocks(wst, n, batch, chunk, crop):
    """Several images in one call, whole and cropped, with chunks that cut images: each equals
    the oracle's image of its own visibilities."""
    fov, n_w, W, per = 0.1, 2, 7, 1500
    img_n = crop or n
    rng = np.random.default_rng([n, batch])
    u, v, w = synth.disk_uvw(batch * per, 0.4 * img_n / fov, 150.0, rng)
    vis = synth.random_visibilities(batch * per, rng)
    off = [i * per for i in range(batch)] + [batch * per]
    cfg, ocfg = config(wst, img_n, fov, n_w, W, planes_per_chunk=chunk, batch=batch, grid_n=n if crop else 0)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis), None, off)
    img = plan.image(flags=wst.WST_NO_CORRECTION).cpu().numpy()
    for i in range(batch):
        s = slice(off[i], off[i + 1])
        ref = oracle.image_on_grid(ocfg, n, u[s], v[s], w[s], vis[s], None, correct=False)
        assert np.abs(img[i] - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("n,W,per_cell", [(64, 8, 1), (256, 3, 5), (512, 8, 64), (1024, 5, 33), (4096, 8, 16)])
def test_table_gradient_with_shared_samples(wst, n, W, per_cell):
    """From one sample per cell (neighbouring taps add to the same sample) up, and supports
    with and without an instance of their own; many visibilities on few cells."""
    fov, n_w, n_vis = 0.1, 2, 4000
    rng = np.random.default_rng([n, W])
    u, v, w, vis = coords("cluster", n, fov, n_vis, rng)
    L = W * per_cell + 1
    xs = np.linspace(-W / 2, W / 2, L)
    tab = (np.exp(-xs**2 / 1.7) * (1 + 0.05 * np.sin(xs))).astype(np.float32)
    cfg = wst.Config(n=n, fov=fov, n_w=n_w, w_min=-160.0, w_max=160.0, support=W, kernel=wst.WST_KERNEL_TABLE,
                     ktable_len=L)
    plan = wst.Plan(cfg)
    plan.set_kernel_table(dev(tab))
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    ocfg = OracleConfig(n, fov, n_w, -160.0, 160.0, W, "table", 0.0, tab.astype(np.float64))
    y = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    got = plan.kernel_grad(dev(y[None])).cpu().numpy()
    ref = oracle.kernel_grad(ocfg, u, v, w, vis, y)
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("n", [2048, 8192])
@pytest.mark.parametrize("n_w,chunk", [(16, 0), (17, 0), (32, 0), (33, 0), (33, 16), (20, 7)])
def test_plane_sum_by_anchor_blocks(wst, n, n_w, chunk):
    """The plane sum where the planes of an image in one call make one, two or more anchor
    blocks of 16, whole and in chunks that cut them, at sampled pixels of the corrected
    image's central half (64- and 128-line tiles)."""
    fov, n_vis, n_pix = 0.1, 400, 48
    rng = np.random.default_rng([n, n_w, chunk])
    u, v, w = synth.disk_uvw(n_vis, 0.45 * n / fov, 150.0, rng)
    vis = synth.random_visibilities(n_vis, rng)
    cfg, ocfg = config(wst, n, fov, n_w, 7, planes_per_chunk=chunk)
    plan = wst.Plan(cfg)
    plan.set_vis(dev(u), dev(v), dev(w), dev(vis))
    img = plan.image()[0].cpu().numpy()
    pa, pb = rng.integers(n // 4, 3 * n // 4, (2, n_pix)).astype(np.int32)
    ref = oracle.image_pixels(ocfg, u, v, w, vis, pa, pb)
    assert np.abs(img[pb, pa] - ref).max() <= TOL * np.abs(ref).max()
