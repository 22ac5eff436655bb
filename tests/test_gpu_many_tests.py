"""More coverage tests than 2^32 in an image small enough to keep its coverage masks in one region:
the count of the tests is exact and the stored masks are not handed out a second time."""
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

W = H = 96
N = 470_000      # fans whose bounds hold the whole image: N W H = 4.33e9 tests


def _frames(n, seen):
    """n fans of four thin triangles along two sides of a square around the image (their bounds cover it,
    their triangles lie outside), then `seen` small fans inside it."""
    cam = synthetic.make_camera((0.0, 0.0, 3.0), W, H)
    half = 3.0 * (W / 2) / cam.fx
    frame = half * np.array([[-1.3, -1.3], [-1.3, 1.3], [-1.4, -1.4], [1.3, -1.3], [-1.4, -1.41]])
    rng = np.random.default_rng(5)
    at = half * rng.uniform(-0.8, 0.8, (seen, 1, 2))
    a = 2 * np.pi * np.arange(4) / 4
    small = at + np.r_[[[0.0, 0.0]], 0.05 * half * np.c_[np.cos(a), np.sin(a)]]
    xy = np.concatenate([np.broadcast_to(frame, (n, 5, 2)), small]).reshape(-1, 2)
    xyz = np.c_[xy, np.repeat(np.r_[np.zeros(n), np.linspace(0.1, 0.2, seen)], 5)].astype(np.float32)
    return cam, xyz, rng.uniform(0, 1, (len(xyz), 3)).astype(np.float32), rng.uniform(0.2, 0.6, len(xyz)).astype(np.float32)


def test_more_than_2_to_32_tests():
    seen = 300
    cam, xyz, rgb, a = _frames(0, seen)
    r = ms.Renderer(seen, 4, cam, ms.render_params(tile=32))
    want = r.forward(dev(xyz), dev(rgb), dev(a)).clone()
    few = r.last_info
    assert few.frags > seen
    _, xyz, _, _ = _frames(N, seen)
    fill = lambda t: np.concatenate([np.full((5 * N,) + t.shape[1:], 0.5, np.float32), t])
    b = ms.Renderer(N + seen, 4, cam, ms.render_params(tile=32, pair_capacity=9 * N + 9 * seen))
    img = b.forward(dev(xyz), dev(fill(rgb)), dev(fill(a)))
    assert b.last_info.rect_tests == N * W * H + few.rect_tests
    assert b.last_info.frags == few.frags
    assert torch.equal(img, want)
