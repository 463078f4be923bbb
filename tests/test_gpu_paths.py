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
