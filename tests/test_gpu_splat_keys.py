"""Depth keys of source Gaussians seen edge-on: splats on one plane through almost the camera centre have equal
FP64 depths along a pixel column, so their index decides the order; the double-float depths must give way to
FP64 wherever their own error could round them to another key."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synthetic  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_07754_gb300._lib as L
    L.lib()


from gpu_util import dev, err_report  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402

W, H, F, CX = 32768, 8, 1000.0, 30000.0


def _scene(planes, each, seed):
    """`planes` planes x = h (h 0.002 to 0.02 from the camera's axis), `each` splats on every one: a plane's
    depths, h F / (px - CX), and so its keys, are the same for all of its splats, exactly."""
    rng = np.random.default_rng(seed)
    cam = synthetic.make_camera((0.0, 0.0, 8.0), W, H)
    cam.fx = cam.fy = F
    cam.cx, cam.cy = CX, H / 2
    n = planes * each
    h = np.repeat(rng.uniform(0.002, 0.02, planes), each)
    means = np.c_[h, rng.uniform(-0.01, 0.01, n), 8.0 - rng.uniform(2.0, 5.0, n)].astype(np.float32)
    ls = np.c_[np.full(n, -12.0), np.log(rng.uniform(0.2, 0.6, (n, 2)))].astype(np.float32)
    q = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1))
    sh = rng.normal(0, 0.9, (n, 1, 3)).astype(np.float32)
    # far apart in opacity between neighbours in index, so that a wrong order shows
    return cam, synthetic.Scene(means, ls, q, rng.uniform(0.02, 0.15, n).astype(np.float32), sh, 0)


@pytest.mark.parametrize("planes,each,tile", [(40, 30, 8), (40, 30, 16), (60, 20, 32)])
def test_order_of_coplanar_splats_seen_edge_on(planes, each, tile):
    for seed in range(6):
        cam, sc = _scene(planes, each, seed)
        rgb = oracle.gaussian_colors(sc).astype(np.float32)
        win = (int(CX) - 8, 0, int(CX) + 24, H)
        ref, nf = oracle.splat_render(sc, cam, rgb=rgb.astype(np.float64), window=win)
        assert nf.max() > 20
        p = ms.render_params(tile=tile, T_eps=1e-30)
        sr = ms.SplatRenderer(sc.n, [cam], p)
        flat = sr.render(dev(sc.means), dev(sc.log_scales), dev(sc.quats), dev(sc.opacity), dev(rgb))
        img = sr.images(flat)[0][:, win[0]:win[2]].cpu().numpy().astype(np.float64)
        rep = err_report(img, ref, 1e-5)
        assert rep["n_over_tol"] == 0, (seed, rep)
