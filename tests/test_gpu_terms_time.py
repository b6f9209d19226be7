"""The optional force terms cost the FP32 walk no more than an eighth of its time."""
import time

import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


def test_terms_against_none():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    n, side = 32768, 32
    k = np.arange(n)
    x = 1.99e-3 * (np.stack([k % side, k // side % side, k // side ** 2], 1) + 0.6)     # six contacts each
    z, r = np.zeros((n, 3)), np.full(n, 1e-3, np.float32)
    base = scenes.drum(seed=1, n=500, precision="fp32", stiffness="hertz").params
    p = base.copy(walls=[], g=(0.0, 0.0, 0.0), domain_lo=(0.0,) * 3, domain_hi=(0.066,) * 3,
                  cell_size=scenes.auto_cell_size(float(r[0])))
    configs = (p, p.copy(terms=15, mu_roll=0.02, alpha_t=0.2, k_coh=2e3))

    def ratio():
        stream = torch.cuda.Stream()
        sims = [dem.Simulation(q, x, z, z, r, cuda_stream=stream.cuda_stream) for q in configs]
        best = [np.inf, np.inf]
        for _ in range(10):
            for j, s in enumerate(sims):
                dem.dem_set_particles(s.h, x, z, z, r)   # (the same contacts every time)
                s.step(4)
                t0 = time.perf_counter()
                s.step(60)
                best[j] = min(best[j], time.perf_counter() - t0)
        for s in sims:
            s.close()
        return best[1] / best[0]

    # (a busy host can slow a whole window: three attempts)
    assert any(ratio() <= 1.125 for _ in range(3))
