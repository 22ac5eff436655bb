"""Shadows in scenes of any scale: the binary32 filter's products round in units of 2^-149 in very small scenes, and
what they no longer decide is left to FP64."""
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


@pytest.mark.parametrize("scale", [1e6, 1.0, 1e-12, 3e-14, 1.5e-14])
def test_shadows_at_a_scale(scale):
    rng = np.random.default_rng(8)
    n = 6000
    c = rng.uniform(-1, 1, (n, 1, 3))
    xyz = (scale * (c + rng.normal(0, 0.03, (n, 3, 3)))).astype(np.float32).reshape(-1, 3)
    tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    rgb = rng.uniform(0, 1, (3 * n, 3)).astype(np.float32)
    a = rng.uniform(0.2, 0.6, 3 * n).astype(np.float32)
    cam = synthetic.make_camera((0.3, 0.4, 3.0), 24, 20)
    cam.C = (np.asarray(cam.C) * scale).astype(np.float32).astype(np.float64)
    cam.znear = float(np.float32(0.01 * scale))
    light = (np.array([2.0, -1.5, 2.5]) * scale).astype(np.float32).astype(np.float64)
    rt = ms.RayTracer(n)
    X, I = dev(xyz), dev(tris)
    rt.build(X, I)
    img = rt.trace(X, dev(rgb), dev(a), cam, tris=I, light=light, ambient=0.2).cpu().numpy()
    ref = ort.render(xyz, rgb, a, tris, cam, light=light, ambient=0.2)
    plain = ort.render(xyz, rgb, a, tris, cam)
    assert np.abs(plain - ref).max() > 0.1        # the light does cast shadows
    assert np.abs(img - ref).max() <= 1e-5
