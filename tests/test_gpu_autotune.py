"""The autotuner times a tile once: its two kbuf values render the same way and report the same figures."""
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


from gpu_util import dev, oracle_mesh_f32  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402


def test_a_tile_is_timed_once():
    n, K = 2000, 8
    soup = [dev(t) for t in oracle_mesh_f32(synthetic.surface_scene(n, 3, degree=0), K)]
    cams = [synthetic.make_camera((0.3, 0.5, 3.2), 80, 60), synthetic.make_camera((2.0, 0.5, 2.2), 64, 64)]
    br = ms.BatchRenderer(n, K, cams)
    res = br.autotune(*soup, reps=3)
    t = list(res.cand_ms)
    assert t[0::2] == t[1::2] and min(t) > 0
    assert list(res.cand_ws_bytes)[0::2] == list(res.cand_ws_bytes)[1::2]
    assert res.best in (0, 2, 4) and res.best_ms == min(t) and br.params.kbuf == 8
