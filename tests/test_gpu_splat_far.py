"""Source Gaussians far from the origin seen from close by: the binary32 vertices of their polygons are off by
a good part of a pixel there, and the splats' outermost centres still lie within the polygons' rectangles."""
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


def scene(at, n, seed):
    """n small splats about one unit in front of a camera (f = 1000 px) at `at`."""
    rng = np.random.default_rng(seed)
    cam = synthetic.make_camera((0.0, 0.0, 4.0), 96, 64)
    cam.fx = cam.fy = 1000.0
    cam.cx, cam.cy = 48.0, 32.0
    cam.C = np.asarray(at, np.float32).astype(np.float64)
    z = rng.uniform(0.8, 1.25, n)
    v = np.c_[rng.uniform(-46, 46, n) / 1000 * z, rng.uniform(-30, 30, n) / 1000 * z, z]
    means = (cam.C + v @ np.asarray(cam.R_cw, np.float64).reshape(3, 3)).astype(np.float32)
    ls = np.c_[np.log(rng.uniform(0.2, 1.5, (n, 2)) / 2700), np.full(n, -12.0)].astype(np.float32)
    q = rng.normal(0, 0.3, (n, 4)) + np.array([1.0, 0, 0, 0])
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    sh = rng.normal(0, 0.8, (n, 1, 3)).astype(np.float32)
    return cam, synthetic.Scene(means, ls, q, rng.uniform(0.2, 0.6, n).astype(np.float32), sh, 0)


@pytest.mark.parametrize("at,tile", [((4000.0, -3500.0, 2500.0), 16), ((4000.0, -3500.0, 2500.0), 8), ((30.0, 1e-3, -20.0), 32),
                                     ((-60000.0, 100.0, 50000.0), 16)])
def test_splats_far_from_the_origin(at, tile):
    cam, sc = scene(at, 20_000, 3)
    rgb = oracle.gaussian_colors(sc).astype(np.float32)
    ref, nf = oracle.splat_render(sc, cam, rgb=rgb.astype(np.float64))
    sr = ms.SplatRenderer(sc.n, [cam], ms.render_params(tile=tile, T_eps=1e-30))
    flat = sr.render(dev(sc.means), dev(sc.log_scales), dev(sc.quats), dev(sc.opacity), dev(rgb))
    rep = err_report(sr.images(flat)[0].cpu().numpy().astype(np.float64), ref)
    print(rep, sr.last_info.frags, int(nf.sum()))
    assert rep["n_over_tol"] == 0, rep
    assert sr.last_info.frags == int(nf.sum())
