"""The source-Gaussian render's coefficients lie in parts of the workspace that a forward render leaves unused
where they fit: the images do not depend on the place, and the workspace is no larger than the fans' and the polygons."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synthetic  # noqa: E402

import paper_2502_07754_gb300 as ms  # noqa: E402
from paper_2502_07754_gb300 import _lib  # noqa: E402


def _sizes(n, cams, p):
    cs = (_lib.Camera * len(cams))(*[ms.camera_struct(c) for c in cams])
    L = _lib.lib()
    return (L.ms_splat_workspace_size(n, cs, len(cams), C.byref(p)), L.ms_batch_workspace_size(n, 8, cs, len(cams), C.byref(p)))


def _cams(views):
    return [synthetic.make_camera((0.2 * v, 0.1, 3.0), 41, 30) for v in range(views)]


# the records hold the coefficients; the gradients do; neither does
@pytest.mark.parametrize("n,views,frags,own", [(20_000, 16, 2_000_000, 0), (20_000, 3, 100, 0), (20_000, 4, 100, 1)])
def test_workspace_size(n, views, frags, own):
    p = ms.render_params()
    p.frag_capacity = frags
    size, fans = _sizes(n, _cams(views), p)
    up = lambda x: (x + 255) // 256 * 256
    assert size == fans + up(n * 9 * 12) + own * up(80 * n * views)


@pytest.mark.gpu
@pytest.mark.parametrize("views", [1, 3, 4])
def test_images_do_not_depend_on_the_place(views):
    from gpu_util import dev
    n = 4000
    rng = np.random.default_rng(views)
    args = [dev(t.astype(np.float32)) for t in (
        rng.normal(0, 0.4, (n, 3)), np.c_[rng.uniform(-5.5, -4.5, (n, 2)), np.full(n, -12.0)],
        rng.normal(0, 1, (n, 4)), rng.uniform(0.2, 0.6, n), rng.uniform(0, 1, (n, 3)))]
    cams = _cams(views)
    p = ms.render_params()
    p.frag_capacity = 4_000_000
    a = ms.SplatRenderer(n, cams, p)
    img = a.render(*args).clone()
    frags = a.last_info.frags
    assert 0 < 32 * frags < 80 * n * views      # (exactly these records do not hold the coefficients)
    q = ms.render_params()
    q.frag_capacity = frags
    b = ms.SplatRenderer(n, cams, q)
    assert torch.equal(b.render(*args), img)
