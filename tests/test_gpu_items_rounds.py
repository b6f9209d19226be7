"""FP64 contact items over several steps with springs, in blocks that take every pair inside once,
in blocks with too many candidates for that and in blocks with too many items: against slabs, which
evaluate every pair from both sides (walk, the same bits), and lists against the walk."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu

BLOCK, ENTRIES, ITEMS = 128, 1280, 768     # a block of the walk and what one of its rounds holds


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    dem.lib()


def _scene(**law):
    """A jittered lattice whose radii grow with z, so that spheres have from 6 contacts to 18."""
    n, side, a = 40000, 34, 1.5e-3
    k = np.arange(n)
    grid = np.stack([k % side, k // side % side, k // side ** 2], 1)
    x = a * (grid + 0.7) + 0.1 * a * scenes.uniform(4, 3 * n, -1.0, 1.0).reshape(n, 3)
    r = (0.85e-3 + 0.3e-3 * grid[:, 2] / grid[:, 2].max()).astype(np.float32)
    v = 0.1 * scenes.uniform(5, 3 * n, -1.0, 1.0).reshape(n, 3)
    w = 5.0 * scenes.uniform(6, 3 * n, -1.0, 1.0).reshape(n, 3)
    base = scenes.drum(seed=4, n=500, precision="fp64").params
    p = base.copy(walls=[], domain_lo=(0.0,) * 3, domain_hi=(a * (side + 1),) * 3,
                  cell_size=scenes.auto_cell_size(float(r.max())))
    return p.copy(**law), x, v, w, r


def _rounds(order, pairs):
    """Blocks of the walk with (entries over the limit, items over the limit with pairs once)."""
    place = np.empty(len(order), np.int64)
    place[order] = np.arange(len(order))
    a, b = place[pairs[:, 0]] // BLOCK, place[pairs[:, 1]] // BLOCK
    blocks = len(order) // BLOCK + 1
    entries = np.bincount(a, minlength=blocks) + np.bincount(b, minlength=blocks)
    items = entries - np.bincount(a[a == b], minlength=blocks)
    return (entries > ENTRIES).sum(), ((entries <= ENTRIES) & (items > ITEMS)).sum(), (items <= ITEMS).sum()


@pytest.mark.parametrize("law", [{}, dict(stiffness="hertz"), dict(terms=15, mu_roll=0.05, alpha_t=0.2, k_coh=1e3)])
def test_walk_against_slabs(law):
    args = _scene(**law)
    with dem.Simulation(*args, max_contacts=64) as s:
        s.forces()
        _, order, pairs = s.snapshot()
        assert min(_rounds(order, pairs)) > 10
        s.step(6)
        want, hist = s.state(), s.history()
    assert len(hist) > 150000
    with dem.Slabs(*args, nslabs=3, max_contacts=64) as z:
        z.step(6)
        for a, b in zip(want, z.state()):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("law", [{}, dict(stiffness="hertz"), dict(model="simple")])
def test_lists_against_the_walk(law):
    # sums over a particle's contacts run in another order: 18 forces of up to 10 N round at 1e-16
    # of them, which moves a sphere of 1e-5 kg by 3e-15 m/s per step of 1.4 us
    p, *arrays = _scene(**law)
    skin = 0.1e-3
    got = []
    for q in (p, p.copy(resort_interval=0, skin=skin, cell_size=p.cell_size + skin)):
        with dem.Simulation(q, *arrays, max_contacts=64) as s:
            if q is not p:
                assert dem.dem_debug_tiles(s.h)[0] == BLOCK
            s.step(6)
            got.append((*s.state(), s.history()))
    (x, v, w, h), (x2, v2, w2, h2) = got
    assert np.max(np.abs(x - x2)) <= 1e-15 and np.max(np.abs(v - v2)) <= 1e-11 and np.max(np.abs(w - w2)) <= 1e-8
    assert np.array_equal(h["i"], h2["i"]) and np.array_equal(h["j"], h2["j"])
    assert len(h) == 0 or np.max(np.abs(h["d"] - h2["d"])) <= 1e-15
