"""Ray tracing where the fast intersection tests are not certain: rays through shared vertices and
along shared edges (closed edges: every triangle that owns the point counts), grazing shadow
segments, degenerate triangles, and sizes around the 8 x 8 pixel blocks -- against the FP64 oracle."""
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


def _camera(w, h):
    """At (0, 0, 4) looking down -z with focal length 64: the rays meet z = 0 at multiples of 1/16 plus 1/32."""
    c = synthetic.make_camera((0.0, 0.0, 4.0), w, h)
    c.fx = c.fy = 64.0
    c.cx, c.cy = 16.0, 16.0
    return c


def _grid(n, cell, z, seed):
    """n x n cells of two triangles each, vertices at odd multiples of 1/32 (on the rays), plus one degenerate triangle."""
    k = np.arange(n + 1) - n // 2
    xy = np.stack(np.meshgrid(k, k, indexing="ij"), -1).reshape(-1, 2) * cell + 1.0 / 32.0
    v = np.c_[xy, np.full(len(xy), z)].astype(np.float32)
    at = lambda i, j: i * (n + 1) + j
    t = []
    for i in range(n):
        for j in range(n):
            t += [(at(i, j), at(i + 1, j), at(i, j + 1)), (at(i + 1, j), at(i + 1, j + 1), at(i, j + 1))]
    t.append((0, 1, 1))
    rng = np.random.default_rng(seed)
    return v, np.asarray(t, np.int32), rng.uniform(0, 1, (len(v), 3)).astype(np.float32), rng.uniform(0.1, 0.5, len(v)).astype(np.float32)


@pytest.mark.parametrize("w,h,cell,light", [(32, 32, 0.125, None), (33, 23, 0.0625, None), (7, 8, 0.25, None),
                                            (32, 32, 0.125, (0.03125, 0.03125, 3.0)), (17, 25, 0.25, (2.0, 0.0, 0.01))])
def test_rays_through_vertices_and_edges(w, h, cell, light):
    v0, t0, c0, a0 = _grid(6, cell, 0.0, 1)
    v1, t1, c1, a1 = _grid(4, cell, 0.25, 2)
    v, c, a = np.r_[v0, v1], np.r_[c0, c1], np.r_[a0, a1]
    t = np.r_[t0, t1 + len(v0)].astype(np.int32)
    cam = _camera(w, h)
    rt = ms.RayTracer(len(t))
    X, T = dev(v), dev(t)
    rt.build(X, T)
    img = rt.trace(X, dev(c), dev(a), cam, tris=T, light=light, ambient=0.25 if light else 1.0).cpu().numpy()
    ref = ort.render(v, c, a, t, cam, light=np.asarray(light, np.float64) if light else None, ambient=0.25 if light else 1.0)
    assert ref[..., 3].max() > 0.1
    assert np.abs(img - ref).max() <= 1e-4
    assert rt.status()[1] == 0


@pytest.mark.parametrize("layers,light", [(24, None), (25, None), (70, None), (16, (0.5, 0.25, 3.0)), (53, (0.5, 0.25, 3.0))])
def test_many_crossings_per_pixel(layers, light):
    """As many crossings as a pass keeps, one more, and several passes; a pixel next to one without any."""
    parts = [_grid(2, 0.125, -0.01 * i, 5 + i) for i in range(layers)]
    v = np.concatenate([p[0] for p in parts])
    v[:, :2] += 0.003   # off the rays: no crossing lies on an edge
    t = np.concatenate([p[1] + i * len(parts[0][0]) for i, p in enumerate(parts)]).astype(np.int32)
    c = np.concatenate([p[2] for p in parts])
    a = np.concatenate([p[3] for p in parts]) * np.float32(0.1)
    cam = _camera(19, 21)
    rt = ms.RayTracer(len(t))
    X, T = dev(v), dev(t)
    rt.build(X, T)
    img = rt.trace(X, dev(c), dev(a), cam, tris=T, light=light, ambient=0.25 if light else 1.0).cpu().numpy()
    ref = ort.render(v, c, a, t, cam, light=np.asarray(light, np.float64) if light else None, ambient=0.25 if light else 1.0)
    assert ref[..., 3].max() > 0.3
    assert np.abs(img - ref).max() <= 1e-4
    assert rt.status()[1] == 0
