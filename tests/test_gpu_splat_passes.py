"""The source-Gaussian render's binary32 / double-float passes at the edges of their range:
sub-pixel and image-sized splats, planes nearly edge-on to the camera, elongated axes, every tile
size, more hits at a pixel than one warp's round takes -- images against the FP64 oracle."""
import math

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


def _scene(n, seed, lo, hi, tilt):
    """n flat Gaussians around the origin, in-plane scales exp(U[lo, hi]); tilt: how far their
    normals turn from the view axis (pi / 2: edge-on)."""
    rng = np.random.default_rng(seed)
    means = rng.normal(0, 0.25, (n, 3)).astype(np.float32)
    ls = np.c_[np.full(n, -12.0), rng.uniform(lo, hi, (n, 2))].astype(np.float32)
    phi = rng.uniform(0, 2 * math.pi, n)
    ax = np.c_[np.cos(phi), np.sin(phi), np.zeros(n)]           # turn axis in the image plane
    z = np.broadcast_to([0.0, 0.0, 1.0], (n, 3))
    ang = tilt * rng.uniform(0.98, 1.0, n)[:, None]
    nrm = z * np.cos(ang) + np.cross(ax, z) * np.sin(ang)
    psi = rng.uniform(0, 2 * math.pi, n)[:, None]
    t2 = np.cross(nrm, ax)
    r2 = np.cos(psi) * ax + np.sin(psi) * t2
    R = np.stack([nrm, r2, np.cross(nrm, r2)], axis=2)
    q = synthetic.scenes.rotmat_to_quat(R).astype(np.float32)
    sh = np.zeros((n, 1, 3), np.float32)
    sh[:, 0, :] = rng.normal(0, 0.8, (n, 3))
    return synthetic.Scene(means, ls, q, rng.uniform(0.05, 0.6, n).astype(np.float32), sh, 0)


@pytest.mark.parametrize("n,lo,hi,tilt,tile", [(1, -1.5, -1.0, 0.5, 16), (33, -5.0, -4.0, 0.8, 8), (300, -3.0, -1.0, 1.0, 16),
                                               (200, -4.0, -0.7, 1.55, 32), (120, -6.0, -0.7, 1.5707, 8),
                                               (400, -1.5, -1.0, 0.3, 16)])
def test_splat_passes_match_oracle(n, lo, hi, tilt, tile):
    sc = _scene(n, 17 + n, lo, hi, tilt)
    cams = [synthetic.make_camera((0.02, 0.03, 3.0), 71, 45), synthetic.make_camera((1.5, 0.4, 2.4), 32, 64)]
    rgb = oracle.gaussian_colors(sc).astype(np.float32)
    sr = ms.SplatRenderer(n, cams, ms.render_params(tile=tile, T_eps=1e-30))
    flat = sr.render(dev(sc.means), dev(sc.log_scales), dev(sc.quats), dev(sc.opacity), dev(rgb))
    for img, cam in zip(sr.images(flat), cams):
        ref, _ = oracle.splat_render(sc, cam, rgb=rgb.astype(np.float64))
        rep = err_report(img.cpu().numpy().astype(np.float64), ref)
        assert rep["n_over_tol"] == 0, rep
