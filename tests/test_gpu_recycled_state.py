"""Saved states are recycled within their context: a state made from a
destroyed one renders as a new one does (larger and smaller scenes, another
stream while the earlier work is in flight, two-round lists), reads as empty
before its first forward, and may be destroyed after its context."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402


def _scene(seed, n, w, h):
    sc = scenes.random_scene(seed, n, [scenes.pinhole(w, h, f=float(w)), scenes.pinhole(h, w, f=float(w))], 1)
    return P.params_of(sc), to_camera_views(sc.views, P.device())


def _images(r, params, cams, saved=None):
    rgb, depth, alpha, saved = r.forward(params, cams, saved=saved)
    return [t.clone() for t in (rgb, depth, alpha)], saved


@pytest.mark.parametrize("no_sync,prefix", [(False, 1.0), (True, 1.0), (False, 0.3)])
def test_recycled_states_render_as_new_ones(no_sync, prefix):
    batches = [_scene(1, 300, 40, 30), _scene(2, 4000, 90, 70), _scene(3, 50, 17, 23), _scene(4, 6000, 64, 64)]
    want = []
    for params, cams in batches:
        r = Rasterizer(sh_degree=1, device=P.device())
        want.append(_images(r, params, cams)[0])
    r = Rasterizer(sh_degree=1, device=P.device())
    r.set_config(list_prefix=prefix)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    got, handles = [], set()
    for i in range(8):
        params, cams = batches[i % 4]
        if no_sync and i >= 4:
            r.set_config(no_sync=True)
        with torch.cuda.stream(streams[i % 2]):
            saved = r.new_saved()
            assert saved.info()["n_pixels"] == 0 and saved.info()["n_visible"] == 0
            handles.add(saved.h.value)
            images, _ = _images(r, params, cams, saved)
            r.backward(params, cams, saved, torch.ones_like(images[0]))
        got.append(images)
        del saved   # its work may still be in flight
    torch.cuda.synchronize()
    assert len(handles) <= 2   # the states were recycled
    for i, images in enumerate(got):
        for a, b in zip(images, want[i % 4]):
            assert torch.equal(a, b)


def test_destroy_order_and_exports():
    params, cams = _scene(5, 200, 32, 24)
    r = Rasterizer(sh_degree=1, device=P.device())
    _, saved = _images(r, params, cams)
    first = saved.h.value
    r.debug_lists(saved)           # read on any stream: not recycled
    del saved
    kept = r.new_saved()
    _images(r, params, cams, kept)
    h, kept.h = kept.h, None
    r.lib.gsr_destroy(r.ctx)       # the context first, then its state
    r.ctx = None
    r.lib.gsr_saved_destroy(h)
    assert first is not None and isinstance(h, C.c_void_p)
    torch.cuda.synchronize()
