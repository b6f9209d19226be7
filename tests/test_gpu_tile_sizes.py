"""Every tile size that large runs use, stepped through several sorts: the same bits whatever the
tile, with halos that fit, that fit in some tiles and in none, on both sides of full tiles, and
for FP64's two sizes."""
import numpy as np
import pytest

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


def _bed(n, precision, skin, speed=0.2):
    sc = scenes.drum(seed=9, n=n, precision=precision)
    v = sc.v + speed * scenes.uniform(10, 3 * n, -1.0, 1.0).reshape(n, 3)
    p = sc.params.copy(resort_interval=0, skin=skin, cell_size=sc.params.cell_size + skin)
    return p, sc.x * 0.998, v, sc.w, sc.r


def _run(args, steps, block=0):
    with dem.Simulation(*args, block_size=block) as s:
        s.step(steps)
        d = s.diagnostics()
        return dem.dem_debug_tiles(s.h), d["sorts"], (*s.state(), s.history(), *s.forces())


def _equal(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("n,skin,want", [(70003, 0.1e-3, {128, 224, 320, 512}), (136009, 0.1e-3, {128, 224, 320, 448}),
                                         (136009, 1.7e-3, {128, 224, 320, 448}),
                                         (155603, 0.1e-3, {128, 224, 320, 512})])
def test_fp32_sizes(n, skin, want):
    """want: the sizes of a GPU of 152 SMs for block sizes 32, 64, 96 and 128."""
    args = _bed(n, "fp32", skin, speed=1e4 * skin)
    first, seen, direct, fit = None, set(), 0, 0
    for block in (32, 64, 96, 128):
        (tile, tiles, none), sorts, out = _run(args, 120, block)
        assert tiles == -(-n // tile) and sorts >= 3
        seen.add(tile)
        direct, fit = direct + none, fit + tiles - none
        first = first or out
        assert _equal(first, out)
    assert seen <= want and len(seen) >= 3, seen
    if skin > 1e-3:
        assert direct > 0 and fit > 0             # both ways of reading partners


@pytest.mark.parametrize("law", [dict(stiffness="hertz"), dict(terms=15, mu_roll=0.02, alpha_t=0.2, k_coh=2e3),
                                 dict(model="simple")])
def test_fp32_sizes_of_every_law(law):
    p, *rest = _bed(136009, "fp32", 0.3e-3)
    runs = [_run((p.copy(**law), *rest), 40, block) for block in (32, 64, 128)]
    assert len({r[0][0] for r in runs}) == 3
    assert _equal(runs[0][2], runs[1][2]) and _equal(runs[0][2], runs[2][2])


@pytest.mark.parametrize("precision,n", [("fp32", 136100), ("fp64", 60000)])
@pytest.mark.parametrize("off", [-1, 0, 1])
def test_around_full_tiles(precision, n, off):
    with dem.Simulation(*_bed(n, precision, 0.2e-3)) as s:
        tile = dem.dem_debug_tiles(s.h)[0]
    assert tile >= 128
    k = n // tile * tile + off
    args = _bed(n, precision, 0.2e-3)
    args = (args[0], *(a[:k] for a in args[1:]))
    big, _, out = _run(args, 30)
    assert big[0] == tile and big[1] == -(-k // tile)
    if precision == "fp32":
        small, _, ref = _run(args, 30, 32)
        assert small[0] < tile and _equal(out, ref)


def test_fp64_sizes():
    """A scene of 30,000 spheres by itself takes tiles of 64, two of them in one batch 128."""
    p, *arrays = _bed(30011, "fp64", 0.1e-3, speed=1.0)
    (tile, _, _), sorts, out = _run((p, *arrays), 60)
    assert tile == 64 and sorts >= 2
    q = p.copy(mu=0.1)
    b = dem.dem_batch_create(precision="fp64")
    slots = [dem.dem_batch_add(b, w, *arrays, 60) for w in (p, q)]
    dem.dem_batch_run(b, 60)
    got = dem.dem_batch_get_state(b, slots[0], 30011)
    dem.dem_batch_destroy(b)
    assert _equal(out[:3], got)
