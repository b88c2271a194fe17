"""Device memory of recycled states: a state that has grown does not make the
context's buffers grow again."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402

MB = 1 << 20


def test_reuse_allocates_nothing():
    # 2000 Gaussians over most of a 1080p view: 16 M instances in 0.14 M tile rows
    dev = P.device()
    sc = scenes.random_scene(6, 2000, [scenes.pinhole(1920, 1080, f=900.0)], 0, z_range=(2.0, 3.0), xy_half=0.5,
                             log_scale_range=(0.0, 0.5))
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    r = Rasterizer(sh_degree=0, device=dev)
    out = tuple(torch.empty(k * 1920 * 1080, device=dev) for k in (3, 1, 1))
    saved = r.new_saved()
    r.forward(params, cams, saved=saved, out=out)
    assert saved.info()["n_instances"] > 4_000_000
    want = [t.clone() for t in out]
    del saved
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    saved = r.new_saved()
    r.forward(params, cams, saved=saved, out=out)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 8 * MB
    for a, b in zip(out, want):
        assert torch.equal(a, b)
