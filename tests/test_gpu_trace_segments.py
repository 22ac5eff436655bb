"""Segments to the light that pass an edge closer than a double-float origin resolves: the FP64 test that
decides them starts from the FP64 point of the crossing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synthetic  # noqa: E402
from oracle import raytrace as ort  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_07754_gb300._lib as L
    L.lib()


from gpu_util import dev  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402

W, H = 16, 400


def _scene():
    """A floor at z = 0 seen from straight above, and a blocker in the plane z = 1 that ends at y = y_e, under a
    light at z = 2: a segment from (x, y, 0) meets the plane half way, at (y + y_light) / 2. With y = h + l + e (its
    double-float parts and the rest), y_light = -l and y_e = h / 2 it misses the edge by e / 2; a row of pixels
    with the largest e > 0 is taken."""
    cam = synthetic.make_camera((0.0, 0.0, 4.0), W, H)
    cam.fx = cam.fy = float(np.float32(371.3))
    cam.cx, cam.cy = W / 2, H / 2
    R = np.asarray(cam.R_cw, np.float64).reshape(3, 3)
    rows = np.arange(H)
    y = 4.0 * R[1, 1] * ((rows + 0.5 - cam.cy) / cam.fy)
    h = y.astype(np.float32)
    low = (y - h).astype(np.float32)
    e = (y - h) - low
    e_rel = np.where(y > 0.2, e / y, -1.0)
    r = int(np.argmax(e_rel))
    # (powers of two: depth 4, the points and the edge's values are exact in FP64, in any order of operations)
    floor = np.array([[-4, -4, 0], [12, -4, 0], [-4, 12, 0]], np.float32)
    blocker = np.array([[-8, h[r] / 2, 1], [8, h[r] / 2, 1], [0, -8, 1]], np.float32)
    xyz = np.r_[floor, blocker]
    return cam, r, e_rel[r], xyz, np.array([[0, 1, 2], [3, 4, 5]], np.int32), (0.0, float(-low[r]), 2.0)


def test_segments_that_miss_an_edge_by_less_than_double_float_resolves():
    cam, r, e_rel, xyz, tris, light = _scene()
    assert e_rel > 2.0 ** -50
    rgb = np.full((6, 3), 0.5, np.float32)
    alpha = np.full(6, 0.5, np.float32)
    rt = ms.RayTracer(2)
    X, I = dev(xyz), dev(tris)
    rt.build(X, I)
    img = rt.trace(X, dev(rgb), dev(alpha), cam, tris=I, light=light, ambient=0.25).cpu().numpy()
    ref = ort.render(xyz, rgb, alpha, tris, cam, light=np.asarray(light, np.float64), ambient=0.25, window=(0, r - 3, W, r + 4))
    assert np.abs(ref[3, :, 0] - 0.25).max() < 1e-12       # the row's segments all miss the blocker
    assert np.abs(img[r - 3:r + 4] - ref).max() <= 1e-6
