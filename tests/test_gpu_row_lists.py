"""Tile lists made by tile rows (batches of 65536 records and 4096 tiles and more): the lists
of small and large records over ragged views and every tile shape against the
oracle, images equal to those of the same views in smaller batches (lists by
sorted instances), two rounds equal to one, and growth from tiny buffers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_2512_08498_gb300 import _lib as L  # noqa: E402
from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402

N = 24_000


def _scene(tile, log_scale=(-6.0, -2.0)):
    views = [scenes.pinhole(203, 77, f=150.0),
             scenes.pinhole(64, 130, f=90.0, viewmat=scenes.look_from([0.2, 0.0, -0.3], yaw_deg=9.0)),
             scenes.pinhole(1, 1, f=2.0), scenes.pinhole(33, 17, f=40.0, viewmat=scenes.look_from([0.0, 0.1, 0.0], roll_deg=30.0)),
             # more than 4096 tiles, empty: it looks away
             scenes.pinhole(1040, 1040, f=500.0, viewmat=scenes.look_from([0.0, 0.0, 0.0], yaw_deg=180.0))]
    return scenes.random_scene(11, N, views, 0, log_scale_range=log_scale, tile=tile)


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("log_scale", [(-6.0, -3.0), (-4.0, -0.5)])
def test_lists_against_the_oracle(tile, log_scale):
    sc = _scene(tile, log_scale)
    assert N * len(sc.views) >= 65536
    o = oracle.Oracle(sc, tile=tile)
    g = P.run_gpu(sc, tile=tile)
    P.compare_lists(g, o, check_reach=log_scale[1] < -1.0)
    # one view at a time: fewer than 65536 records, so the lists are sorted instances
    offs = np.cumsum([0] + [v.width * v.height for v in sc.views])
    for i, v in enumerate(sc.views):
        one = scenes.Scene(sc.name, sc.means, sc.log_scales, sc.quats, sc.opacity_logits, sc.sh, 0, [v], tile=tile, bg=sc.bg)
        g1 = P.run_gpu(one, tile=tile)
        assert np.array_equal(g1["rgb"], g["rgb"][3 * offs[i]:3 * offs[i + 1]])
        assert np.array_equal(g1["ncontrib"], g["ncontrib"][offs[i]:offs[i + 1]])


@pytest.mark.parametrize("prefix", [0.03, 0.3, 0.9])
def test_two_rounds_and_growth(prefix):
    sc = _scene((16, 16), (-4.0, -0.5))
    dev = P.device()
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    images = []
    for f in (1.0, prefix, 0.0):
        r = Rasterizer(sh_degree=0, device=dev)
        r.set_config(list_prefix=f)
        saved = r.new_saved()
        r.lib.gsr_reserve(r.ctx, saved.h, 1, 1)   # grows the buffers and renders again
        for _ in range(2):
            out = r.forward(params, cams, saved=saved)[:3]
        grads = r.backward(params, cams, saved, torch.ones_like(out[0]) / out[0].numel())
        images.append([t.clone() for t in out] + list(r.debug_pixels(saved)) + list(grads))
    for other in images[1:]:
        for k, (a, b) in enumerate(zip(images[0], other)):
            if k < 5:
                assert torch.equal(a, b), k
            else:
                # the order of the backward's atomic additions
                assert float((a - b).norm()) <= 1e-6 * float(a.norm()), k


def test_timeout_skips_the_row_lists():
    # an earlier kernel's wait gives up: the lists' kernels skip their work, the
    # call reports it, and the next one renders
    sc = _scene((16, 16))
    dev = P.device()
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    r = Rasterizer(sh_degree=0, device=dev)
    want = [t.clone() for t in r.forward(params, cams)[:3]]
    r.debug_set_wait(wait_ns=200_000, withhold_prefix=True)
    with pytest.raises(L.GsrError) as e:
        r.forward(params, cams)
    assert e.value.code == L.GSR_ERR_TIMEOUT
    r.debug_set_wait(0, False)
    for a, b in zip(want, r.forward(params, cams)[:3]):
        assert torch.equal(a, b)
