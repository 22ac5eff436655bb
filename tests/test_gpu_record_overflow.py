"""A fragment buffer that is too small: the overflow is reported, and every pixel of the image is written --
with what it holds in full where its records fit, with the background where they do not.  Fragments are
counted in 64 bits however many there are."""
import ctypes as C

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


from gpu_util import dev, oracle_mesh_f32  # noqa: E402
import paper_2502_07754_gb300 as ms  # noqa: E402
from paper_2502_07754_gb300 import _lib  # noqa: E402


# room for 1 record, for less than one span of 1024 pixels, and for half of the scene's
@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("room", [1, 1000, 0.5])
def test_every_pixel_is_written(tile, room):
    n, K = 6000, 8
    sc = synthetic.surface_scene(n, 11, degree=0)
    cam = synthetic.make_camera((0.3, 0.5, 3.2), 96, 80)
    soup = [dev(t) for t in oracle_mesh_f32(sc, K)]
    bg = (0.125, 0.25, 0.5)
    p = ms.render_params(tile=tile, bg=bg, T_eps=1e-30)
    full = ms.Renderer(n, K, cam, p)
    want = full.forward(*soup).clone()
    frags = full.last_info.frags
    p.frag_capacity = int(room * frags) if room < 1 else room
    cs = ms.camera_struct(cam)
    L = _lib.lib()
    nbytes = L.ms_render_workspace_size(n, K, C.byref(cs), C.byref(p))
    ws = torch.full((nbytes + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    wsp = C.c_void_p(ws.data_ptr() + (256 - ws.data_ptr() % 256) % 256)
    out = torch.full((cam.height, cam.width, 4), -7.0, device="cuda")
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert L.ms_render(*[C.c_void_p(t.data_ptr()) for t in soup], n, K, C.byref(cs), C.byref(p), C.c_void_p(out.data_ptr()),
                       wsp, nbytes, stream) == _lib.MS_OK
    info = _lib.RenderInfo()
    assert L.ms_render_get_info(wsp, C.byref(info), stream) == _lib.MS_ERR_CAPACITY
    assert info.overflow == 1 and info.frags == frags
    is_bg = (out == torch.tensor([*bg, 0.0], device="cuda")).all(-1)
    is_full = (out == want).all(-1)
    assert bool((is_bg | is_full).all())
    held = int((is_full & ~is_bg).sum())
    assert held > 100 if room == 0.5 else held <= room


def test_more_than_2_to_32_fragments_of_one_span():
    """4.3M fans over an image of one 32 x 32 tile: every centre lies in one triangle of each."""
    n, K = 4_300_000, 3
    cam = synthetic.make_camera((0.0, 0.0, 3.0), 32, 32)
    half = 3.0 * 16 / cam.fx
    fan = half * np.array([[0.01, 0.013, 0], [8.0, 0.3, 0], [-5.0, 7.0, 0], [-4.5, -6.5, 0]])
    xyz = torch.tensor(fan.astype(np.float32), device="cuda").repeat(n, 1)
    rgb = torch.full_like(xyz, 0.5)
    a = torch.full((len(xyz),), 0.25, device="cuda")
    p = ms.render_params(tile=32, bg=(0.125, 0.25, 0.5), pair_capacity=n)
    r = ms.BatchRenderer(n, K, [cam], p)
    flat = r.forward(xyz, rgb, a, flat=r.new_flat(-7.0), check_status=False)
    st, info = r.info()
    assert st == _lib.MS_ERR_CAPACITY and info.pairs == n
    assert info.frags == n * 1024 > info.frag_capacity
    assert bool((flat == torch.tensor([0.125, 0.25, 0.5, 0.0], device="cuda")).all())
