"""Rays order their crossings by FP64 depths: two planes closer than double-float numbers resolve, the
nearer one drawn in front although its triangles come last."""
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


@pytest.mark.parametrize("gap", [3e-15, 1e-12, 1e-6])
def test_planes_closer_than_double_float_resolves(gap):
    """gap 3e-15 at a depth of 3.4 is 7 units of FP64's last place, and half a unit of a double-float's."""
    quad = np.array([[-3.1, -2.9, 0], [3.3, -3.2, 0], [2.9, 3.4, 0], [-3.2, 3.0, 0]], np.float32)
    near = quad + np.array([0, 0, gap], np.float32)
    xyz = np.r_[quad, near]
    tris = np.array([[0, 1, 2], [0, 2, 3], [4, 5, 6], [4, 6, 7]], np.int32)
    rgb = np.repeat(np.array([[0, 1, 0], [1, 0, 0]], np.float32), 4, axis=0)
    alpha = np.full(8, 0.5, np.float32)
    cam = synthetic.make_camera((1.3, 0.7, 3.1), 40, 36)
    rt = ms.RayTracer(4)
    X, I = dev(xyz), dev(tris)
    rt.build(X, I)
    img = rt.trace(X, dev(rgb), dev(alpha), cam, tris=I).cpu().numpy()
    ref = ort.render(xyz, rgb, alpha, tris, cam)
    seen = ref[..., 3] > 0     # (the planes end inside the image)
    assert seen.mean() > 0.9 and np.abs(ref[seen] - np.array([0.5, 0.25, 0.0, 0.75])).max() <= 1e-12   # the oracle resolves them
    assert np.abs(img - ref).max() <= 1e-6
