"""The list build around the particle counts where its warps take 4, 8, 16 or 32 positions: the
contact pairs are those of the 27-cell walk."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [3, 19455, 19457, 38911, 38913, 77823, 77825])
def test_pairs_of_the_walk(n, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    sc = scenes.drum(seed=17, n=n, precision=precision)
    x, skin = sc.x * 0.998, 0.1e-3
    got = []
    for p in (sc.params, sc.params.copy(resort_interval=0, skin=skin, cell_size=sc.params.cell_size + skin)):
        with dem.Simulation(p, x, sc.v, sc.w, sc.r) as s:
            s.forces()
            got.append(s.snapshot()[2])
    assert np.array_equal(*got)
    assert n < 10 or len(got[0]) > n // 2          # (the bed has about n contacts)
