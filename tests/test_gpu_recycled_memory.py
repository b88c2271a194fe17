"""Device memory of recycled states: a state that has grown does not make the
context's buffers grow again, and the kept states are given back to every call whose
own allocation fails."""
import numpy as np
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


def test_kept_states_are_given_back_to_other_calls():
    dev = P.device()
    n = 3_000_000
    rng = np.random.default_rng(1)
    sc = scenes.random_scene(6, 4, [scenes.pinhole(64, 64, f=60.0)], 0)
    params = [torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(dev) for a in (
        np.stack([rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.uniform(2, 6, n)], 1), np.full((n, 3), -7.0),
        np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)), np.zeros(n), np.zeros((n, 1, 3)))]
    r = Rasterizer(sh_degree=0, device=dev)
    r.forward(params, to_camera_views(sc.views, dev))   # (its state, about 400 MB, is destroyed and kept)
    images = [(torch.rand(3 * 1600 * 900, device=dev), 1600, 900, 1)] * 18
    x = torch.empty(18, device=dev)
    r.dft_energy(images[:1], out=x[:1])                 # plans and tables
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.cuda.mem_get_info()[0] - 96 * MB
    block = torch.empty(room, dtype=torch.uint8, device=dev)
    try:
        # 18 half spectra of 17 MB do not fit beside the block
        assert torch.cuda.mem_get_info()[0] < 18 * 17 * MB
        r.dft_energy(images, out=x)
        torch.cuda.synchronize()
    finally:
        del block
        torch.cuda.empty_cache()
    assert torch.equal(x, x[:1].expand(18))
