"""The backward's sums over a warp's pixels: the moments about the centre of
an 8x4 pixel block, shifted to the record's mean, and which pixels share them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402

U = 2.0 ** -24   # half an ulp, relative


@pytest.mark.parametrize("batch", [128, 256, 512])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
def test_second_moment_of_records_on_one_corner_pixel(tile, batch):
    # 256 records of opacity 0.01 and the low-pass footprint, each on one corner
    # pixel of an 8x8 block (0.01 exp(-0.5 0.9^2 / 0.3) < 1/255: no neighbour
    # composites), up to 0.1 pixel off its centre
    at = np.array([x for b in range(8) for x in (8 * b, 8 * b + 7)])
    px, py = (a.reshape(-1) for a in np.meshgrid(at, at))
    rng = np.random.default_rng(5)
    u, v = px + 0.5 + rng.uniform(-0.1, 0.1, 256), py + 0.5 + rng.uniform(-0.1, 0.1, 256)
    sc = scenes.random_scene(3, 256, [scenes.pinhole(64, 64, f=64.0)], 0, tile=tile)
    sc.means[:] = np.stack([(u - 32.0) * 2.0 / 64.0, (v - 32.0) * 2.0 / 64.0, np.full(256, 2.0)], 1)
    sc.log_scales[:] = -9.0
    sc.opacity_logits[:] = np.log(0.01 / 0.99)
    dev = P.device()
    r = Rasterizer(tile=tile, sh_degree=0, device=dev)
    r.set_config(batch_bwd=batch)
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    _, _, _, saved = r.forward(params, cams)
    assert saved.info()["blended_pairs"] == 256
    g = torch.Generator(device=dev)
    g.manual_seed(1)
    r.backward(params, cams, saved, torch.randn(3 * 64 * 64, generator=g, device=dev))
    rec, grec = (t.cpu().numpy().astype(np.float64) for t in (r.debug_records(saved)[0], r.debug_record_grads(saved)))
    # one pixel: dL/dqc = ln2 gP dy^2 with gP = dL/dsigma sigma
    dy = py + 0.5 - rec[:, 1]
    gp = grec[:, 5] * rec[:, 5]
    want = np.log(2.0) * gp * dy * dy
    # roundings of myy - 2 uy my + uy^2 m0 with |yo| = 1.5, |uy| <= 1.6: one each
    # of my (1.5, times 2 uy), myy (2.25), their difference (2.55) and uy^2
    # (2.56); then a few of the small result and of gP
    bound = U * np.log(2.0) * np.abs(gp) * (2 * 1.6 * 1.5 + 2.25 + 2.55 + 2.56) + 8 * U * np.abs(want)
    assert np.all(np.abs(grec[:, 4] - want) <= bound), np.max(np.abs(grec[:, 4] - want) / bound)


@pytest.mark.parametrize("depth", [False, True])
def test_non_finite_colour_stays_with_its_pixel_block(depth):
    # two small Gaussians in one 8x8 pixel block, in its upper and its lower 8x4
    # half: the first one's infinite colour leaves the second's gradients alone
    sc = scenes.random_scene(7, 2, [scenes.pinhole(16, 16, f=20.0)], 0)
    for i, (u, z) in enumerate(((1.5, 3.0), (6.5, 2.0))):
        sc.means[i] = ((u - 8.0) * z / 20.0, (u - 8.0) * z / 20.0, z)
    sc.log_scales[:] = -3.5
    sc.opacity_logits[:] = 1.0
    dev = P.device()
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    up_rgb, up_dep = torch.randn(3 * 256, generator=g, device=dev), torch.randn(256, generator=g, device=dev)
    got = []
    for value in (0.5, np.inf):
        sc.sh[0] = value
        r = Rasterizer(sh_degree=0, bg=sc.bg, device=dev)
        params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
        _, _, alpha, saved = r.forward(params, cams)
        assert float(alpha[17]) > 0.1 and float(alpha[6 * 16 + 6]) > 0.1
        got.append(r.backward(params, cams, saved, up_rgb, up_dep if depth else None)[:5])
    for a, b in zip(*got):
        assert torch.allclose(a[1], b[1], rtol=1e-6, atol=0.0)
