"""Tiles of list mode: every tile size, tiles whose halo does not fit (partners read from
global memory), ragged last tiles, springs set after the lists (restore, in any record
order), against the sort-every-step mode in FP64 and against one another bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    dem.lib()


def _squeezed(n, seed, precision, stiffness="linear"):
    """A drum bed shrunk by 0.2%, so that it starts with contacts."""
    sc = scenes.drum(seed=seed, n=n, precision=precision, stiffness=stiffness)
    sc.x *= 0.998
    sc.v += np.random.default_rng(seed).normal(0.0, 0.2, size=sc.x.shape)
    return sc


def _listed(params, skin):
    return params.copy(resort_interval=0, skin=skin, cell_size=params.cell_size + skin)


@pytest.mark.parametrize("skin", [0.1e-3, 2.2e-3])   # the larger one overflows the small tiles' halos
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tile_sizes_give_the_same_bits(precision, skin):
    sc = _squeezed(5003, 5, precision)
    p = _listed(sc.params, skin)
    got = []
    for block in (32, 64, 96, 128, 256):
        with dem.Simulation(p, sc.x, sc.v, sc.w, sc.r, block_size=block) as s:
            s.step(60)
            got.append((*s.state(), s.history(), s.forces()[0]))
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
    ref = oracle.State(sc.params.copy(precision="fp64"), sc.x, sc.v, sc.w, sc.r).run(60)
    assert np.max(np.abs(got[0][0] - ref.x)) <= (1e-12 if precision == "fp64" else 1e-9)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 511, 512, 513, 1025])
def test_ragged_tiles(n):
    sc = _squeezed(2000, 6, "fp64", "hertz")
    x, v, w, r = sc.x[:n], sc.v[:n], sc.w[:n], sc.r[:n]
    with dem.Simulation(_listed(sc.params, 0.2e-3), x, v, w, r) as s:
        s.step(40)
        a = s.state()
    ref = oracle.State(sc.params, x, v, w, r).run(40)
    assert np.max(np.abs(a[0] - ref.x)) <= 1e-12


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_restored_springs_in_any_order(precision):
    sc = _squeezed(3001, 7, precision)
    p = _listed(sc.params, 0.1e-3)
    with dem.Simulation(p, sc.x, sc.v, sc.w, sc.r) as s:
        s.step(30)
        st, h = s.state(), s.history()
        s.step(50)
        want = s.state()
    assert len(h) > 1000
    for order in (np.arange(len(h)), np.random.default_rng(1).permutation(len(h))):
        with dem.Simulation(p, sc.x, sc.v, sc.w, sc.r) as s:
            dem.dem_restore(s.h, *st, sc.r, h[order])
            s.step(50)
            for a, b in zip(want, s.state()):
                assert np.array_equal(a, b)
