"""Batches of many small scenes in list mode: the tiles follow the scenes, not their total."""
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


def _scene(n, seed, precision):
    sc = scenes.drum(seed=seed, n=max(n, 600), precision=precision)
    skin = 0.2e-3
    p = sc.params.copy(resort_interval=0, skin=skin, cell_size=sc.params.cell_size + skin)
    v = 0.1 * scenes.uniform(seed + 1, 3 * n, -1.0, 1.0).reshape(n, 3)
    return p, sc.x[:n] * 0.998, v, sc.w[:n], sc.r[:n]


def _batch(sizes, precision, seeds):
    b = dem.dem_batch_create(precision=precision)
    slots = [dem.dem_batch_add(b, *_scene(n, s, precision), 1000) for n, s in zip(sizes, seeds)]
    return b, slots


def test_small_scenes_take_small_tiles():
    """50 times as many scenes of 64 spheres take no more than 50 times the memory: with a tile
    for their total every scene would hold the halo of a tile of hundreds."""
    got = []
    for k in (20, 1000):
        b, _ = _batch([64] * k, "fp32", [3 + j % 5 for j in range(k)])
        dem.dem_batch_run(b, 1)
        got.append(dem.dem_batch_device_bytes(b))
        dem.dem_batch_destroy(b)
    assert got[1] <= 50 * got[0]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes", [[64] * 600, [33, 97, 161, 193] * 80, [1, 31, 700] * 60, [90] * 400 + [20000]])
def test_each_scene_keeps_the_bits_of_its_own_run(sizes, precision):
    seeds = [3 + k % 4 for k in range(len(sizes))]
    b, slots = _batch(sizes, precision, seeds)
    dem.dem_batch_run(b, 25)
    own = {}
    for slot, n, seed in zip(slots, sizes, seeds):
        if (n, seed) not in own:
            p, x, v, w, r = _scene(n, seed, precision)
            with dem.Simulation(p, x, v, w, r) as s:
                s.step(25)
                own[n, seed] = s.state()
        for a, c in zip(dem.dem_batch_get_state(b, slot, n), own[n, seed]):
            assert np.array_equal(a, c)
    dem.dem_batch_destroy(b)
