"""Work items beyond one launch: with room for so many items that the raster passes stride over
them, the images are those of a grid with a warp for every item."""
import math

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

W, H = 3000, 3008           # 141,000 tiles of 8 pixels, each with at least one fan: an item or more
CAPACITY = 36_000_000       # pairs: room for 700,000 items, more than the grid has warps


def _params(frags=0, capacity=0):
    p = ms.render_params(tile=8, pair_capacity=capacity)
    p.frag_capacity = frags
    return p


@pytest.mark.parametrize("K", [6, 8, 5])
def test_strided_items_match_one_warp_each(K):
    n = 6
    rng = np.random.default_rng(K)
    c = np.c_[rng.uniform(-0.4, 0.4, (n, 2)), rng.uniform(-0.2, 0.2, n)]
    rad = np.r_[6.0, rng.uniform(0.2, 1.0, n - 1)]
    a = 2 * math.pi * np.arange(K) / K
    ring = np.c_[np.cos(a), np.sin(a), np.zeros(K)]
    xyz = np.concatenate([c[:, None], c[:, None] + rad[:, None, None] * ring], 1).reshape(-1, 3)
    V = n * (K + 1)
    soup = [dev(t.astype(np.float32)) for t in (xyz, rng.uniform(0, 1, (V, 3)), rng.uniform(0.1, 0.6, V))]
    cam = synthetic.make_camera((0.0, 0.0, 3.0), W, H)
    r = ms.Renderer(n, K, cam, _params())
    img = r.forward(*soup).clone()
    inf = r.last_info
    assert inf.pairs >= 141_000
    del r
    s = ms.Renderer(n, K, cam, _params(inf.frags, CAPACITY))
    assert torch.equal(s.forward(*soup), img)
    assert (s.last_info.pairs, s.last_info.frags, s.last_info.rect_tests) == (inf.pairs, inf.frags, inf.rect_tests)


def test_strided_splat_items_match_one_warp_each():
    n = 5
    rng = np.random.default_rng(3)
    means = np.c_[rng.uniform(-0.3, 0.3, (n, 2)), rng.uniform(-0.2, 0.2, n)].astype(np.float32)
    ls = np.c_[np.full((n, 2), -1.2), np.full(n, -9.0)].astype(np.float32)
    ls[0, :2] = 1.2
    q = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1))
    args = [dev(t.astype(np.float32)) for t in (means, ls, q, rng.uniform(0.2, 0.6, n), rng.uniform(0, 1, (n, 3)))]
    cam = synthetic.make_camera((0.0, 0.0, 3.0), W, H)
    a = ms.SplatRenderer(n, [cam], _params())
    img = a.render(*args).clone()
    frags = a.last_info.frags
    assert a.last_info.pairs >= 141_000
    del a
    b = ms.SplatRenderer(n, [cam], _params(frags, CAPACITY))
    assert torch.equal(b.render(*args), img)
