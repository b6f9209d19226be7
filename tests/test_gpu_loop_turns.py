"""Step counts and forced sort intervals around the turn lengths of the step loop: odd counts stay
in the loop, and the bits are those of plain launches."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    return torch.cuda.Stream()


def _scene(interval, speed):
    sc = scenes.drum(seed=12, n=1501, precision="fp32")
    v = speed * scenes.uniform(13, 3 * 1501, -1.0, 1.0).reshape(1501, 3)
    skin = 0.2e-3
    return sc, v, sc.params.copy(resort_interval=interval, skin=skin, cell_size=sc.params.cell_size + skin)


@pytest.mark.parametrize("k", [2, 3, 7, 11, 13, 20, 33, 47])
def test_every_step_of_a_call_is_three_launches(stream, k):
    sc, v, p = _scene(0, 0.0)
    with dem.Simulation(p, sc.x, v, sc.w, sc.r, cuda_stream=stream.cuda_stream) as s:
        s.step(k)
        sorts = s.diagnostics()["sorts"]
        before = dem.dem_launch_count(s.h)
        s.step(k)
        launches = dem.dem_launch_count(s.h) - before
        assert s.diagnostics()["sorts"] == sorts     # (slow spheres: none falls due)
        assert launches == 3 * k


@pytest.mark.parametrize("interval", [0, 2, 3, 7, 11])
def test_counts_and_intervals_against_plain_launches(stream, interval):
    sc, v, p = _scene(interval, 1.0)
    calls = (3, 5, 11, 12, 13, 23, 47, 4, 1, 6)
    got = []
    for st, split in ((None, (sum(calls),)), (stream.cuda_stream, calls)):
        with dem.Simulation(p, sc.x, v, sc.w, sc.r, cuda_stream=st) as s:
            for n in split:
                s.step(n)
            d = s.diagnostics()
            got.append((*s.state(), s.history(), d["sorts"], d["steps"]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_scenes_join_a_batch_after_an_odd_number_of_steps(stream, precision):
    """The springs of the scenes that stay are taken from the buffer the last step wrote."""
    sc, v, p = _scene(0, 0.3)
    p = p.copy(precision=precision)
    b = dem.dem_batch_create(precision=precision, cuda_stream=stream.cuda_stream)
    slots = [dem.dem_batch_add(b, p, sc.x, v, sc.w, sc.r, 1000)]
    for k in (7, 3, 12):
        dem.dem_batch_run(b, k)
        slots.append(dem.dem_batch_add(b, p, sc.x, v, sc.w, sc.r, 1000))
    dem.dem_batch_run(b, 9)
    got = [dem.dem_batch_get_state(b, s, 1501) for s in slots]
    dem.dem_batch_destroy(b)
    for out, steps in zip(got, (31, 24, 21, 9)):
        with dem.Simulation(p, sc.x, v, sc.w, sc.r) as s:
            s.step(steps)
            for a, c in zip(out, s.state()):
                assert np.array_equal(a, c)
