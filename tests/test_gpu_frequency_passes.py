"""The transform's passes: every composite radix alone and combined, prime
passes before them, single-pass lengths, and both layouts of a call (few
columns: one channel per row item and one column per column item; many: three
and four), against the oracle within the norm-wise FFT bound."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machines
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_frequency import _check, _raster  # noqa: E402

SIZES = [(2, 3), (4, 5), (6, 8), (9, 10), (12, 15), (16, 1), (1, 16), (18, 20), (45, 60), (96, 144), (33, 77), (112, 99),
         (49, 22), (241, 36), (1201, 24), (150, 1922)]


@pytest.mark.parametrize("many", [False, True])
def test_every_radix(many):
    rng = np.random.default_rng(9)
    imgs = [rng.random((3, h, w)) for h, w in SIZES]
    if many:
        # enough columns for the wide layouts (8 per SM)
        imgs += [rng.random((3, 7, 640)) for _ in range(5)]
        _check(_raster(), imgs, [1] * len(imgs))
    else:
        r = _raster()
        for img in imgs:
            _check(r, [img], [1])
    _check(_raster(), imgs, [3] * len(imgs))
