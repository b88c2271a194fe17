"""The blends walk a tile's list in chunks of 32 entries per 8x8 pixel block,
the backward its composited entries in groups of eight: list lengths around
those edges, pixels that stop inside a chunk, image edges inside a block, and
records whose form is too ill-conditioned for the culling threshold, against
the oracle."""
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


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("n,logit", [(1, 0.0), (2, 2.0), (31, -2.0), (32, -2.0), (33, -2.0), (64, 0.0), (65, -3.0),
                                     (97, 3.0)])
def test_list_lengths(n, logit, tile):
    # every Gaussian covers the whole 21 x 13 image; n is each tile's list length
    views = [scenes.pinhole(21, 13, f=20.0), scenes.pinhole(9, 17, f=20.0)]
    sc = scenes.random_scene(40 + n, n, views, 1, z_range=(2.0, 4.0), xy_half=0.3, log_scale_range=(-0.6, 0.2), tile=tile,
                             bg=(0.2, 0.1, 0.4))
    sc.opacity_logits[:] = logit
    if n > 4:
        # a needle (condition above 1e5 after the low-pass) among them
        sc.log_scales[n // 2] = (2.5, -7.0, -7.0)
    o = oracle.Oracle(sc, tile=tile)
    ref = o.forward()
    up_o, up_g = P.upstream(sc, o, ref)
    g = P.run_gpu(sc, tile=tile, grads=up_g)
    P.compare_lists(g, o)
    P.compare_pixels(g, o, ref)
    P.compare_counters(g, o, ref, with_bwd=True)
    P.compare_images(g, ref)


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("depth", [False, True])
@pytest.mark.parametrize("n,logit", [(1, 0.0), (7, -1.0), (8, -1.0), (9, -1.0), (16, 5.5), (31, -2.0), (32, -2.0),
                                     (33, -2.0), (40, -2.5), (65, -3.0), (97, 3.0)])
def test_backward_groups(n, logit, depth, tile):
    # n entries that every pixel may composite (all of them at low opacity;
    # at logit 5.5 the 0.99 clamp acts), with and without a depth gradient
    views = [scenes.pinhole(21, 13, f=20.0), scenes.pinhole(9, 17, f=20.0)]
    sc = scenes.random_scene(70 + n, n, views, 1, z_range=(2.0, 4.0), xy_half=0.3, log_scale_range=(-2.0, -0.5), tile=tile,
                             bg=(0.2, 0.1, 0.4))
    sc.opacity_logits[:] = logit
    o = oracle.Oracle(sc, tile=tile)
    ref = o.forward()
    up_o, up_g = P.upstream(sc, o, ref, depth_w=0.05 if depth else 0.0)
    dev = P.device()
    r = Rasterizer(tile=tile, sh_degree=1, bg=sc.bg, device=dev)
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    _, _, _, saved = r.forward(params, cams)
    d_rgb, d_dep, d_alp = (torch.from_numpy(x).to(dev) for x in up_g)
    grads = r.backward(params, cams, saved, d_rgb, d_dep if depth else None, d_alp, want_focal=True)
    g = dict(info=saved.info(), grec=r.debug_record_grads(saved).cpu().numpy(),
             grads={k: t.cpu().numpy().astype(np.float64) for k, t in zip(P.PARAM_NAMES + ["pose", "focal"], grads)})
    assert g["info"]["bwd_pairs"] > 0
    go = o.backward(up_o[0], up_o[1], up_o[2], want_grec=True)
    P.compare_grads(g, go)
    P.compare_record_grads(g, go)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("depth", [False, True])
def test_non_finite_upstream_gradient_stays_with_its_pixel(depth, bad):
    # two small Gaussians in one 8x8 block; only the first reaches the pixel
    # (1, 1), so the second's gradients are those of a zero there
    sc = scenes.random_scene(7, 2, [scenes.pinhole(16, 16, f=20.0)], 0)
    for i, u in enumerate((1.5, 6.5)):
        sc.means[i] = ((u - 8.0) * 2.0 / 20.0, (u - 8.0) * 2.0 / 20.0, 2.0)
    sc.log_scales[:] = (-5.0, -3.5, -3.0)
    sc.opacity_logits[:] = 1.0
    dev = P.device()
    r = Rasterizer(sh_degree=0, bg=sc.bg, device=dev)
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    _, _, alpha, saved = r.forward(params, cams)
    assert float(alpha[17]) > 0.1 and float(alpha[6 * 16 + 6]) > 0.1
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    up_rgb, up_dep = torch.randn(3 * 256, generator=g, device=dev), torch.randn(256, generator=g, device=dev)
    got = []
    for value in (0.0, bad):
        d_rgb, d_dep = up_rgb.clone(), up_dep.clone()
        d_rgb[17] = d_dep[17] = value
        got.append(r.backward(params, cams, saved, d_rgb, d_dep if depth else None)[:5])
    for a, b in zip(*got):
        # the same terms but for the exponential's rounding (16 ulp at most, 1e-6),
        # in sums that cancel to no less than a hundredth
        assert torch.allclose(a[1], b[1], rtol=1e-4, atol=1e-4 * float(a[1].abs().max()))
    assert not bool(torch.isfinite(got[1][4][0]).all())
