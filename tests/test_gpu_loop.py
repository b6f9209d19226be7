"""The step loop of list mode (a graph that sorts by itself when the device decides to)
against plain launches: any split of the steps into calls, forced sorts, and a step that
is voided by a contact-slot overflow inside the loop."""
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


def _scene(precision, interval):
    sc = scenes.drum(seed=12, n=3001, precision=precision)
    v = np.random.default_rng(12).normal(0.0, 1.0, size=sc.x.shape)
    skin = 0.1e-3
    return sc, v, sc.params.copy(resort_interval=interval, skin=skin, cell_size=sc.params.cell_size + skin)


@pytest.mark.parametrize("interval", [0, 5])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_loop_equals_plain_launches_for_any_split(stream, precision, interval):
    sc, v, p = _scene(precision, interval)
    calls = (2, 3, 7, 8, 9, 1, 16, 17, 30, 33)
    got = []
    for st, split in ((None, (sum(calls),)), (stream.cuda_stream, calls), (stream.cuda_stream, (sum(calls),))):
        with dem.Simulation(p, sc.x, v, sc.w, sc.r, cuda_stream=st) as s:
            for k in split:
                s.step(k)
            d = s.diagnostics()
            got.append((*s.state(), s.history(), d["sorts"], d["steps"], d["pair_contacts"], d["max_overlap"]))
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
    assert got[0][4] > 3


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_overflow_inside_the_loop_is_redone(stream, precision):
    sc, v, p = _scene(precision, 0)
    got = []
    for slots in (2, 32):
        with dem.Simulation(p, sc.x, v, sc.w, sc.r, cuda_stream=stream.cuda_stream, max_contacts=slots) as s:
            s.step(41)
            s.step(10)
            got.append((*s.state(), s.history(), s.diagnostics()["steps"]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
