"""Tile lists and pixel record ranges at their edges: more tiles than one block of the tile scan
takes, one-pixel and one-row images, a pair list that fits exactly, empty scenes and tiles, work
items of every size -- the image does not depend on any of them."""
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


from gpu_util import dev, err_report, oracle_mesh_f32, oracle_render  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402


@pytest.mark.parametrize("n,w,h", [(3000, 331, 259), (40, 1, 1), (500, 1, 200), (2000, 513, 16), (1, 64, 64), (20000, 96, 96)])
def test_image_does_not_depend_on_tiles_or_capacities(n, w, h):
    K = 8
    sc = synthetic.surface_scene(n, 300 + n, degree=0)
    cam = synthetic.make_camera((0.3, 0.5, 3.2), w, h)
    soup = oracle_mesh_f32(sc, K)
    X, Cc, A = (dev(t) for t in soup)
    ref, _, _ = oracle_render(*soup, K, cam)
    base = None
    for tile in (16, 8, 32):
        r = ms.Renderer(n, K, cam, ms.render_params(tile=tile))
        img = r.forward(X, Cc, A)
        assert err_report(img.cpu().numpy().astype(np.float64), ref)["max_abs"] <= 1e-4
        if base is None:
            base = img
        assert torch.equal(img, base)
        # lists that just hold the scene (the work items are then the largest), and one that is twice as long
        for cap in (r.last_info.pairs, 2 * r.last_info.pairs):
            p = ms.render_params(tile=tile, pair_capacity=max(cap, 1))
            p.frag_capacity = max(r.last_info.frags, 1)
            r2 = ms.Renderer(n, K, cam, p)
            assert torch.equal(r2.forward(X, Cc, A), base)
            assert r2.last_info.pairs == r.last_info.pairs and r2.last_info.frags == r.last_info.frags


def test_empty_scene_is_background():
    cam = synthetic.make_camera((0.0, 0.0, 4.0), 37, 21)
    z = torch.zeros(0, 3, device="cuda")
    r = ms.Renderer(0, 8, cam, ms.render_params(bg=(0.25, 0.5, 0.75)))
    img = r.forward(z, z, torch.zeros(0, device="cuda"))
    assert torch.equal(img, torch.tensor([0.25, 0.5, 0.75, 0.0], device="cuda").expand(21, 37, 4))
