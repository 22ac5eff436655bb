"""Binning projects a fan's boundary vertices two at a time: odd and even K, blocks with a
remainder and vertices behind the camera give the oracle's fragments, culled triangles and image."""
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


@pytest.mark.parametrize("n,K,eye", [(257, 3, (0.1, 0.2, 3.0)), (1, 4, (0.0, 0.1, 2.5)), (300, 5, (0.3, -0.2, 2.0)),
                                     (256, 7, (0.1, 0.0, 0.9)), (513, 8, (0.0, 0.2, 0.6)), (100, 15, (0.2, 0.3, 0.7)),
                                     (70, 16, (0.1, 0.1, 2.2))])
def test_fragments_and_image_match_oracle(n, K, eye):
    cam = synthetic.make_camera(eye, 83, 61)
    soup = oracle_mesh_f32(synthetic.surface_scene(n, 70 + n, degree=0), K)
    ref, nf, culled = oracle_render(*soup, K, cam)
    r = ms.Renderer(n, K, cam, ms.render_params(tile=8, T_eps=1e-30))
    img = r.forward(*(dev(t) for t in soup))
    assert err_report(img.cpu().numpy(), ref)["max_abs"] <= 1e-4
    assert r.last_info.frags == int(nf.sum()) and r.last_info.culled_tris == culled
