"""The fill pass of the rasteriser at the edges of its work split: more tests than the count
pass can store masks for (coverage then comes from the decided vertices), items that end inside
a group of staged fans, generic and specialised K, every tile size -- images and gradients
against the FP64 oracle, within the tolerances of the forward and backward parity tests."""
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


from gpu_util import dev, err_report, oracle_mesh_f32, oracle_render  # noqa: E402


def _wide_fans(n, seed, size):
    """n fans facing a camera on the z axis, each about `size` units wide, at separate depths."""
    rng = np.random.default_rng(seed)
    means = np.c_[rng.normal(0, 0.3, (n, 2)), np.linspace(-0.5, 0.5, n)].astype(np.float32)
    q = rng.normal(0, 0.02, (n, 4)) + np.array([math.sqrt(0.5), 0, -math.sqrt(0.5), 0])   # thin axis -> z
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    sh = np.zeros((n, 1, 3), np.float32)
    sh[:, 0, :] = rng.normal(0, 1, (n, 3))
    ls = np.array([[-9, math.log(size), math.log(size)]] * n, np.float32)
    return synthetic.Scene(means, ls, q, rng.uniform(0.02, 0.2, n).astype(np.float32), sh, 0)


# 200 fans over nearly all of 960 pixels: about 190k tests against 80,896 stored masks
@pytest.mark.parametrize("n,K,tile,size", [(200, 8, 16, 0.8), (200, 5, 32, 0.8), (150, 6, 8, 0.8), (33, 8, 16, 0.05),
                                           (1, 16, 16, 0.2), (17, 3, 8, 0.1)])
def test_fill_matches_oracle(n, K, tile, size):
    import paper_2502_07754_gb300 as ms
    cam = synthetic.make_camera((0.05, 0.02, 3.0), 40, 24)
    xyz, rgb, a = oracle_mesh_f32(_wide_fans(n, n + K, size), K)
    orc, nf, _ = oracle_render(xyz, rgb, a, K, cam)
    assert nf.max() >= 1
    r = ms.Renderer(n, K, cam, ms.render_params(tile=tile, T_eps=1e-30))
    X, Cc, A = dev(xyz), dev(rgb), dev(a)
    img = r.forward(X, Cc, A)
    rep = err_report(img.cpu().numpy(), orc)
    assert rep["max_abs"] <= 1e-4, rep
    dL = np.random.default_rng(2).normal(size=orc.shape)
    got = r.backward(X, Cc, A, img, dev(dL.astype(np.float32)))
    want = oracle.render_backward(xyz.astype(np.float64), rgb, a, oracle.fan_tris(n, K), cam, dL.astype(np.float32).astype(np.float64))
    for g, o in zip(got, want):
        o = np.asarray(o)
        assert np.abs(g.cpu().numpy().reshape(o.shape) - o).max() <= 1e-2 * np.abs(o).max() + 1e-6
