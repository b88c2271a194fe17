"""The forward blend's two forms (a warp per 8x8 pixel block, eight warps in step
per tile): the same bits, and which lists take which.  A batch of two views of
797 x 703 has 4400 tiles and may take the first; each view alone, with 2200, takes
the second.  The forms walk different numbers of entries (8x8 blocks against 8x4),
so the statistics tell which one ran."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402

W, H = 797, 703


def _scene(n, hot, tile):
    """n Gaussians spread evenly over both images and `hot` more on one spot."""
    views = [scenes.pinhole(W, H, f=800.0), scenes.pinhole(W, H, f=800.0, viewmat=scenes.look_from([0.02, 0.0, 0.0]))]
    sc = scenes.random_scene(17, n + hot, views, 0, tile=tile, bg=(0.1, 0.2, 0.3))
    rng = np.random.default_rng(4)
    z = rng.uniform(3.0, 5.0, n + hot)
    u, v = rng.uniform(-30.0, W + 30.0, n + hot), rng.uniform(-30.0, H + 30.0, n + hot)
    u[n:], v[n:] = 404.0 + rng.uniform(-3.0, 3.0, hot), 350.0 + rng.uniform(-3.0, 3.0, hot)
    sc.means[:] = np.stack([(u - W / 2) * z / 800.0, (v - H / 2) * z / 800.0, z], 1)
    sc.log_scales[:] = rng.uniform(-4.0, -2.5, (n + hot, 3))
    sc.log_scales[n:] = -6.0
    sc.opacity_logits[:] = rng.uniform(-4.0, 3.0, n + hot)
    return sc


def _render(sc, views, prefix, batch, grads=True):
    dev = P.device()
    r = Rasterizer(tile=sc.tile, batch=batch, sh_degree=0, bg=sc.bg, device=dev)
    r.set_config(list_prefix=prefix)
    params, cams = P.params_of(sc, dev), to_camera_views(views, dev)
    for _ in range(2 if prefix == 0.0 else 1):   # the automatic fraction is chosen by the first forward
        rgb, depth, alpha, saved = r.forward(params, cams)
    tf, nc = r.debug_pixels(saved)
    info = saved.info()
    up = torch.ones_like(rgb) / (3 * W * H)
    g = r.backward(params, cams, saved, up)[:5] if grads else None
    return dict(rgb=rgb, depth=depth, alpha=alpha, tf=tf, nc=nc), info, g


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("hot,prefix,batch", [(0, 1.0, 256), (0, 0.4, 256), (0, 0.0, 256), (6000, 1.0, 256),
                                              (6000, 0.4, 256), (6000, 0.0, 128), (6000, 1.0, 512)])
def test_batch_equals_its_views(tile, hot, prefix, batch):
    sc = _scene(9000, hot, tile)
    both, info, g = _render(sc, sc.views, prefix, batch)
    walked, blended, examined, sums = 0, 0, 0, None
    for i, v in enumerate(sc.views):
        one, info1, g1 = _render(sc, [v], 1.0, batch)
        assert info1["n_tiles"] < 4096 <= info["n_tiles"]
        for k, t in one.items():
            c = 3 if k == "rgb" else 1
            assert torch.equal(both[k][c * i * W * H:c * (i + 1) * W * H], t), k
        walked += info1["warp_entries_fwd"]
        blended += info1["blended_pairs"]
        examined += info1["fwd_pairs"]
        sums = g1 if sums is None else [a + b for a, b in zip(sums, g1)]
    assert info["blended_pairs"] == blended and info["fwd_pairs"] == examined
    for a, b in zip(g, sums):
        # the order of binary32 additions
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
    if prefix == 1.0:
        # the hot spot's list is longer than a resident block's share of the work
        assert (info["warp_entries_fwd"] == walked) == (hot > 0)


@pytest.mark.parametrize("n,batch", [(20_000, 128), (60_000, 128), (60_000, 256)])   # (two rounds pay)
def test_both_forms_choose_the_same_first_round(n, batch):
    # the automatic fraction follows from where the pixels of each tile had stopped,
    # in steps of the staging batch; a view twice (the warp form) has the shares of
    # the view once (the tile form)
    sc = _scene(n, 0, (16, 16))
    sc.opacity_logits[:] = 4.0
    sc.log_scales[:] = np.random.default_rng(1).uniform(-3.0, -2.0, (n, 3))
    one = _render(sc, sc.views[:1], 0.0, batch, grads=False)[1]
    two = _render(sc, [sc.views[0]] * 2, 0.0, batch, grads=False)[1]
    assert one["n_tiles"] < 4096 <= two["n_tiles"]
    assert 0.0 < one["list_prefix"] < 1.0
    assert two["list_prefix"] == one["list_prefix"]


def test_a_replayed_graph_chooses_the_form_again():
    # the same captured forward over even lists, over lists with a hot spot, and over
    # even ones again, its buffers large enough for all
    dev = P.device()
    even, hot = _scene(9000, 6000, (16, 16)), _scene(9000, 6000, (16, 16))
    even.means[9000:] = even.means[:6000]
    even.log_scales[9000:] = even.log_scales[:6000]
    r = Rasterizer(sh_degree=0, bg=even.bg, device=dev)
    cams = to_camera_views(even.views, dev)
    want = []
    for sc in (even, hot):
        params = P.params_of(sc, dev)
        saved = r.new_saved()
        want.append([t.clone() for t in r.forward(params, cams, saved=saved)[:3]] + [saved.info()["warp_entries_fwd"]])
        assert saved.info()["n_tiles"] >= 4096
    held = [t.clone() for t in P.params_of(even, dev)]
    saved = r.new_saved()
    assert r.lib.gsr_reserve(r.ctx, saved.h, 0, 2_000_000) == 0
    out = r.forward(held, cams, saved=saved)[:3]
    r.set_config(no_sync=True)
    r.forward(held, cams, saved=saved, out=out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        r.forward(held, cams, saved=saved, out=out)
    for k in (0, 1, 0):
        for h, p in zip(held, P.params_of((even, hot)[k], dev)):
            h.copy_(p)
        graph.replay()
        torch.cuda.synchronize()
        r.check(saved)
        assert saved.info()["warp_entries_fwd"] == want[k][3]
        for a, b in zip(out, want[k]):
            assert torch.equal(a, b)
