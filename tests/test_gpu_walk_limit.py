"""FP32 walk around the size where a thread per particle takes over from contact items (128
spheres per SM): a sixth more spheres cost no more than a sixth more time."""
import time

import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


def _cube(n, model):
    """A cubic lattice of overlapping spheres at rest (six contacts each, 27 cells full)."""
    k, side = np.arange(n), int(np.ceil(n ** (1 / 3)))
    grid = np.stack([k % side, k // side % side, k // side ** 2], 1)
    x = 1.99e-3 * (grid + 0.6) + 2e-6 * scenes.uniform(31, 3 * n, -1.0, 1.0).reshape(n, 3)
    base = scenes.drum(seed=1, n=500, precision="fp32", model=model).params
    hi = 2e-3 * (side + 1)
    p = base.copy(walls=[], g=(0.0, 0.0, 0.0), domain_lo=(0.0,) * 3, domain_hi=(hi,) * 3,
                  cell_size=scenes.auto_cell_size(float(np.float32(1e-3))))
    z = np.zeros((n, 3))
    return p, x, z, z, np.full(n, 1e-3, np.float32)


@pytest.mark.parametrize("model", ["practical", "simple"])
def test_time_grows_no_faster_than_the_size(model):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    stream = torch.cuda.Stream()
    sizes = (112 * sms, 131 * sms)
    sims = [dem.Simulation(*_cube(n, model), cuda_stream=stream.cuda_stream) for n in sizes]
    best = [np.inf, np.inf]
    for _ in range(25):
        for k, s in enumerate(sims):
            t0 = time.perf_counter()
            s.step(20)
            best[k] = min(best[k], time.perf_counter() - t0)
    for s in sims:
        s.close()
    assert best[1] <= best[0] * sizes[1] / sizes[0]
