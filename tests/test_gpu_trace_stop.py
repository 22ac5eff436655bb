"""Where a shadow segment stops: its transmittance is the product of the factors up to the first that takes it
below T_eps, in the order of the walk -- not of however many the warp had tested by then; and the first crossing
of a ray counts whatever the bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synthetic  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_07754_gb300._lib as L
    L.lib()


from gpu_util import dev  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402

W, H, LAYERS = 48, 40, 12


def _quad(z, x0, x1, y0, y1):
    return np.array([[x0, y0, z], [x1, y0, z], [x1, y1, z], [x0, y1, z]], np.float32)


def _trace(layer_alpha, T_eps, size=1.0):
    """A floor at z = 0 (opacity 0.75, colour 0.5) seen from straight above, `size` of its full extent, which fills
    the view (a small one leaves most lanes of a warp without a segment); beside the view, between the floor
    and a low light, a stack of upright quads of one opacity."""
    cam = synthetic.make_camera((0.0, 0.0, 4.0), W, H)
    v = [_quad(0.0, *(size * np.array([-6, 6.37, -5.83, 6.1])))]   # (no pixel's ray meets its diagonal)
    for i in range(LAYERS):   # planes x = 5 + i / 8, tall enough to cut every segment to the light
        x = 5.0 + i / 8
        v.append(np.array([[x, -9, -1], [x, 9, -1], [x, 9, 9], [x, -9, 9]], np.float32))
    xyz = np.concatenate(v)
    tris = np.concatenate([[[4 * i, 4 * i + 1, 4 * i + 2], [4 * i, 4 * i + 2, 4 * i + 3]] for i in range(LAYERS + 1)]).astype(np.int32)
    alpha = np.r_[np.full(4, 0.75), np.full(4 * LAYERS, layer_alpha)].astype(np.float32)
    rgb = np.full((len(xyz), 3), 0.5, np.float32)
    rt = ms.RayTracer(len(tris))
    X, I = dev(xyz), dev(tris)
    rt.build(X, I)
    return rt.trace(X, dev(rgb), dev(alpha), cam, tris=I, light=(8.0, 0.013, 3.1), ambient=0.25, T_eps=T_eps).cpu().numpy()


@pytest.mark.parametrize("size", [1.0, 0.02])
@pytest.mark.parametrize("layer_alpha,T_eps,factors", [(0.5, 0.3, 2), (0.5, 0.01, 7), (0.25, 0.5, 3), (0.5, 0.0, LAYERS)])
def test_transmittance_stops_at_the_factor_that_blocks(layer_alpha, T_eps, factors, size):
    img = _trace(layer_alpha, T_eps, size)
    seen = img[..., 3] > 0
    assert seen.all() if size == 1.0 else 0 < seen.sum() < 10
    got = (img[seen, 0] / (0.75 * 0.5) - 0.25) / 0.75      # transmittance of every segment
    want = (1.0 - layer_alpha) ** factors
    assert np.abs(got - want).max() <= 1e-6


def test_first_factor_and_first_crossing_count_whatever_the_bound():
    """A bound above 1 ends a composite after its first crossing and a segment after its first factor."""
    img = _trace(0.5, 2.0)
    assert np.abs(img[..., 3] - 0.75).max() <= 1e-6
    assert np.abs((img[..., 0] / (0.75 * 0.5) - 0.25) / 0.75 - 0.5).max() <= 1e-6


def test_images_repeat_bit_for_bit():
    """Blocks hand their segments out in any order; a coarse bound must not let that show."""
    rng = np.random.default_rng(4)
    n = 3000
    xyz = (rng.uniform(-1, 1, (n, 1, 3)) + rng.normal(0, 0.15, (n, 3, 3))).astype(np.float32).reshape(-1, 3)
    tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    X, I = dev(xyz), dev(tris)
    rgb, a = dev(rng.uniform(0, 1, (3 * n, 3)).astype(np.float32)), dev(rng.uniform(0.05, 0.3, 3 * n).astype(np.float32))
    cam = synthetic.make_camera((0.3, 0.4, 3.0), 200, 160)
    rt = ms.RayTracer(n)
    rt.build(X, I)
    first = None
    for _ in range(8):
        img = rt.trace(X, rgb, a, cam, tris=I, light=(2.0, -1.5, 2.5), ambient=0.2, T_eps=0.05)
        first = img.clone() if first is None else first
        assert torch.equal(img, first)
