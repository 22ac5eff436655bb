"""Ray tracing of scenes of no and of one triangle, with and without a light: the background, and the
oracle's image (a tree without an inner node)."""
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


@pytest.mark.parametrize("light", [None, (0.5, 0.5, 3.0)])
@pytest.mark.parametrize("T", [0, 1])
def test_scene_of_no_and_of_one_triangle(T, light):
    xyz = np.array([[-0.7, -0.6, 0.0], [0.8, -0.5, 0.1], [0.1, 0.9, -0.1]], np.float32)
    rgb = np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1]], np.float32)
    alpha = np.array([0.3, 0.6, 0.9], np.float32)
    tris = np.array([[0, 1, 2]], np.int32)[:T]
    cam = synthetic.make_camera((0.1, 0.2, 3.0), 19, 13)
    bg = (0.25, 0.5, 0.75)
    rt = ms.RayTracer(T, K=3)
    X, I = dev(xyz), dev(tris)
    rt.build(X, I if T else None)
    img = rt.trace(X, dev(rgb), dev(alpha), cam, tris=I if T else None, light=light, ambient=0.25 if light else 1.0, bg=bg)
    ref = ort.render(xyz, rgb, alpha, tris, cam, light=np.asarray(light, np.float64) if light else None,
                     ambient=0.25 if light else 1.0, bg=bg)
    assert (ref[..., 3].max() > 0.1) == (T > 0)
    assert np.abs(img.cpu().numpy() - ref).max() <= 1e-5
    if T:
        assert rt.status()[1] == 0


@pytest.mark.parametrize("T", [0, 1])
def test_status_after_a_build(T):
    """The build clears the status word, whatever the memory held before, of an empty scene too."""
    rt = ms.RayTracer(T, K=3)
    rt.bvh.fill_(255)
    xyz = dev(np.array([[-0.7, -0.6, 0.0], [0.8, -0.5, 0.1], [0.1, 0.9, -0.1]], np.float32))
    rt.build(xyz, dev(np.array([[0, 1, 2]], np.int32)[:T]) if T else None)
    assert rt.status() == (0, 0)
