"""Lists by tile rows on views of more than 32 tile columns (not a multiple of 32)
beside a narrow one, every tile shape: a state with room for six million instances
takes them, a fresh one sorts the instances, and everything that a caller reads is
the same.  Small records against the oracle; large ones (runs across columns 32 and
64, chunks of more than 32 runs), in one round and two, against the sorted lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402

N = 33_500


def _scene(tile, log_scale):
    # 65 (16x16), 33 (32x8) or 130 (8x32) tile columns, and 4, 2 or 8
    views = [scenes.pinhole(1040, 1040, f=700.0),
             scenes.pinhole(64, 130, f=90.0, viewmat=scenes.look_from([0.2, 0.0, -0.3], yaw_deg=9.0))]
    sc = scenes.random_scene(12, N, views, 0, z_range=(2.0, 6.0), xy_half=3.0, log_scale_range=log_scale, tile=tile)
    assert N * len(views) >= 65536
    return sc


def _run(sc, rows, prefix=1.0):
    dev = P.device()
    r = Rasterizer(tile=sc.tile, sh_degree=0, bg=sc.bg, device=dev)
    r.set_config(list_prefix=prefix)
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    saved = r.new_saved()
    if rows:
        assert r.lib.gsr_reserve(r.ctx, saved.h, 0, 6_000_000) == 0
    out = r.forward(params, cams, saved=saved)[:3]
    before = r.stats()["launches"]
    r.forward(params, cams, saved=saved, out=out)
    launches = r.stats()["launches"] - before
    keys, vals, ranges = r.debug_lists(saved)
    g = dict(rgb=out[0], depth=out[1], alpha=out[2], keys=keys, vals=vals, ranges=ranges)
    g["tf"], g["nc"] = r.debug_pixels(saved)
    g = {k: t.cpu().numpy() for k, t in g.items()}
    g.update(keys=g["keys"].view(np.uint64), vals=g["vals"].view(np.uint32), ranges=g["ranges"].view(np.uint32),
             info=saved.info())
    return g, launches


def _same(a, b):
    for k in ("n_instances", "n_instances_second", "open_tiles", "n_instances_full", "blended_pairs", "fwd_pairs"):
        assert a["info"][k] == b["info"][k], k
    for k in ("rgb", "depth", "alpha", "tf", "nc"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
def test_lists_against_the_oracle(tile):
    sc = _scene(tile, (-6.0, -3.0))
    g, launches = _run(sc, True)
    s, sorted_launches = _run(sc, False)
    assert launches != sorted_launches   # the two ways
    P.compare_lists(g, oracle.Oracle(sc, tile=tile), check_reach=False)
    _same(g, s)
    for k in ("keys", "vals", "ranges"):
        assert np.array_equal(g[k], s[k]), k


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("prefix", [1.0, 0.05, 0.5])
def test_large_records_against_sorted_instances(tile, prefix):
    sc = _scene(tile, (-4.5, -1.3))
    g, launches = _run(sc, True, prefix)
    s, sorted_launches = _run(sc, False, prefix)
    assert launches != sorted_launches
    if prefix == 1.0 and tile[1] == 8:
        # the most tile rows: more than 8192 chunks of 32 runs, so chunks are longer
        tx = np.array([-(-v.width // tile[0]) for v in sc.views])
        t = (g["keys"] >> np.uint64(32)).astype(np.int64)
        first = tx[0] * -(-sc.views[0].height // tile[1])
        row = np.where(t < first, t // tx[0], 1000 + (t - first) // tx[1])
        assert np.unique(row * (2 * N) + g["vals"]).size > 8192 * 32
    _same(g, s)
    # the regions' starts follow the buffers; each tile's list is the same
    for k in ("keys", "vals"):
        for a, b in zip(g["ranges"][:: max(1, len(g["ranges"]) // 400)], s["ranges"][:: max(1, len(g["ranges"]) // 400)]):
            assert np.array_equal(g[k][a[0]:a[1]], s[k][b[0]:b[1]]), k
    assert np.array_equal(g["ranges"][:, 1] - g["ranges"][:, 0], s["ranges"][:, 1] - s["ranges"][:, 0])


@pytest.mark.parametrize("prefix", [0.05, 0.5])
def test_first_region_of_two_rounds_is_exported_whole(prefix):
    # the first round's lists of the tiles that the second one listed again
    # keep their tile ids
    sc = _scene((16, 16), (-4.5, -1.3))
    g, _ = _run(sc, True, prefix)
    s, _ = _run(sc, False, prefix)
    assert s["info"]["open_tiles"] > 0
    m = s["info"]["n_instances"] - s["info"]["n_instances_second"]
    assert 0 < m and np.array_equal(g["vals"][:m], s["vals"][:m])
    assert np.array_equal(g["keys"][:m], s["keys"][:m])
