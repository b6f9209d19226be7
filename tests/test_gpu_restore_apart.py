"""Springs of pairs that are out of each other's reach: a restored history holds them until the
next step, in list mode as in the walk, and they change nothing."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("resort_interval", [0, 1, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_history_holds_what_was_restored(precision, resort_interval):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    n, skin = 2001, 0.1e-3
    sc = scenes.drum(seed=7, n=n, precision=precision)
    p = sc.params
    if resort_interval != 1:
        p = p.copy(resort_interval=resort_interval, skin=skin, cell_size=p.cell_size + skin)
    with dem.Simulation(p, sc.x * 0.998, sc.v, sc.w, sc.r) as s:
        s.step(30)
        state, near = s.state(), s.history()
        s.step(40)
        want = s.state()
    assert len(near) > 500 and (near["j"] >= dem.WALL_BASE).any()
    # three far partners for every 50th sphere, before, between and behind the near ones
    far = [(i, j) for i in range(0, n - 700, 50) for j in (i + 1, i + 333, i + 690)
           if np.linalg.norm(state[0][i] - state[0][j]) > 6e-3 and not ((near["i"] == i) & (near["j"] == j)).any()]
    assert len(far) > 40
    extra = np.zeros(len(far), dem.HIST_DTYPE)
    extra["i"], extra["j"] = np.array(far).T
    extra["d"] = np.float32(1e-7) * np.arange(3 * len(far)).reshape(-1, 3).astype(np.float32)
    given = np.concatenate([near, extra])
    given = given[np.lexsort((given["j"], given["i"]))]
    with dem.Simulation(p, sc.x, sc.v, sc.w, sc.r) as s:
        dem.dem_restore(s.h, *state, sc.r, given)
        assert np.array_equal(s.history(), given)
        s.step(40)
        for a, b in zip(want, s.state()):
            assert np.array_equal(a, b)
