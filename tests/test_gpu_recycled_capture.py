"""A recycled state whose earlier work was asynchronous, first used inside a CUDA
graph capture: the call waits for that work on the host without ending the capture,
and the replayed graph renders."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2512_08498_gb300 import scenes  # noqa: E402
from paper_2512_08498_gb300.rasterizer import Rasterizer, to_camera_views  # noqa: E402

import _parity as P  # noqa: E402


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_first_forward_of_a_recycled_state_in_a_capture(mode):
    dev = P.device()
    sc = scenes.random_scene(3, 2000, [scenes.pinhole(96, 80, f=90.0)], 1)
    params, cams = P.params_of(sc, dev), to_camera_views(sc.views, dev)
    r = Rasterizer(sh_degree=1, device=dev)
    want = [t.clone() for t in r.forward(params, cams)[:3]]   # (its state is destroyed: buffers of the right sizes)
    r.set_config(no_sync=True)
    saved = r.new_saved()
    first = saved.h.value
    out = r.forward(params, cams, saved=saved)[:3]
    r.backward(params, cams, saved, torch.ones_like(out[0]))
    del saved                                                  # its work was not waited for
    saved = r.new_saved()
    assert saved.h.value == first                              # recycled
    for t in out:
        t.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode=mode):
        r.forward(params, cams, saved=saved, out=out)
    for _ in range(2):
        for t in out:
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        r.check(saved)
        for a, b in zip(out, want):
            assert torch.equal(a, b)
