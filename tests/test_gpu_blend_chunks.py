"""The forward walks a tile's list in chunks of 32 entries per 8x8 pixel
block: list lengths around the chunk edges, pixels that stop inside a chunk,
image edges inside a block, and records whose form is too ill-conditioned for
the culling threshold, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_2512_08498_gb300 import scenes  # noqa: E402

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
