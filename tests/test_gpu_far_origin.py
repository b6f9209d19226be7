"""FP64 walk far from the origin with wide cells: the FP32 prefilter's margin is then many radii
and passes every sphere of the 27 cells, more than a block's round holds. Contacts decide."""
import numpy as np
import pytest

import oracle
from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["practical", "simple"])
@pytest.mark.parametrize("n", [700, 2197])       # below and above the 768 items of a round
def test_many_candidates_few_contacts(n, model):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    r0, at = 1e-3, 1e5
    k = np.arange(2197)
    grid = np.stack([k % 13, k // 13 % 13, k // 169], 1)[:n]
    u = scenes.uniform(21, 3 * n, -1.0, 1.0).reshape(n, 3)
    x = at + 1.99e-3 * (grid + 0.5) + 5e-6 * u                      # lattice neighbours overlap
    v = 0.05 * scenes.uniform(22, 3 * n, -1.0, 1.0).reshape(n, 3)
    w = 5.0 * scenes.uniform(23, 3 * n, -1.0, 1.0).reshape(n, 3)
    r = np.full(n, r0, np.float32)
    base = scenes.drum(seed=1, n=500, precision="fp64", model=model).params
    p = base.copy(walls=[], domain_lo=(at,) * 3, domain_hi=(at + 0.03,) * 3, cell_size=0.02)
    with dem.Simulation(p, x, v, w, r) as s:
        F, _ = s.forces()
        s.step(5)
        got = s.state()
    Fo = oracle.forces(p, x, v, w, r)[0]
    # positions carry 1.5e-11 m of rounding (2^-36 at 1e5 m), times the stiffness per contact
    assert np.max(np.abs(F - Fo)) <= 12 * p.kn * 1.5e-11 + 1e-12
    ref = oracle.State(p, x, v, w, r).run(5)
    assert np.max(np.abs(got[0] - ref.x)) <= 5 * 2 * 1.5e-11
