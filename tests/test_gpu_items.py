"""The force pass by contact items: particle counts around the block sizes it picks, blocks
whose items take more than one round, and the FP32 walk on both sides of its size limit."""
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


def _dense(n, seed, squeeze, **kw):
    """A drum bed shrunk so that spheres overlap: squeeze 0.998 gives a few contacts each,
    0.97 about ten, more than one round of items per block holds."""
    sc = scenes.drum(seed=seed, n=n, **kw)
    sc.x *= squeeze
    sc.v += np.random.default_rng(seed).normal(0.0, 0.1, size=sc.x.shape)
    return sc


def _params(sc, lists):
    if not lists:
        return sc.params
    skin = 0.1e-3
    return sc.params.copy(resort_interval=0, skin=skin, cell_size=sc.params.cell_size + skin)


@pytest.mark.parametrize("lists", [False, True])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 2433, 4865])
def test_block_edges_fp64(n, lists):
    sc = _dense(5000, 3, 0.998, precision="fp64", stiffness="hertz")
    x, v, w, r = sc.x[:n], sc.v[:n], sc.w[:n], sc.r[:n]
    with dem.Simulation(_params(sc, lists), x, v, w, r) as s:
        s.step(20)
        a = s.state()
    ref = oracle.State(sc.params, x, v, w, r).run(20)
    assert np.max(np.abs(a[0] - ref.x)) <= 1e-12


@pytest.mark.parametrize("lists", [False, True])
@pytest.mark.parametrize("model,terms", [("practical", 0), ("practical", 15), ("simple", 0)])
def test_several_rounds_fp64(lists, model, terms):
    # 40,000 particles: blocks of 128, the largest; forces and torques against the oracle
    sc = _dense(40000, 4, 0.97, precision="fp64", model=model)
    p = _params(sc, lists).copy(terms=terms, mu_roll=0.05, alpha_t=0.2, k_coh=1e3)
    with dem.Simulation(p, sc.x, sc.v, sc.w, sc.r, max_contacts=64) as s:
        F, T = s.forces()
    Fo, To = oracle.forces(p, sc.x, sc.v, sc.w, sc.r)[:2]
    S = np.linalg.norm(Fo, axis=1).max()
    assert np.max(np.abs(F - Fo)) <= 1e-11 * S
    assert np.max(np.abs(T - To)) <= 1e-11 * max(np.abs(To).max(), 1e-30)


def test_fp32_walk_across_the_size_limit():
    """The first spheres of one scene with the rest far away: items below 20,000 particles, a
    thread per particle above, the same bits for the same neighbours."""
    sc = _dense(19000, 8, 0.998, precision="fp32")
    far = np.array([sc.params.domain_hi]) * 1.0
    k = 1500
    x2 = np.concatenate([sc.x, far + 4e-3 * (1 + np.arange(k))[:, None]])
    z = np.zeros((k, 3))
    v2, w2 = np.concatenate([sc.v, z]), np.concatenate([sc.w, z])
    r2 = np.concatenate([sc.r, np.full(k, sc.r.min(), np.float32)])
    got = []
    for x, v, w, r in ((sc.x, sc.v, sc.w, sc.r), (x2, v2, w2, r2)):
        p = sc.params.copy(walls=[])
        # (24 slots: the block's lists take exactly the default limit of shared memory)
        with dem.Simulation(p, x, v, w, r, max_contacts=24) as s:
            s.step(20)
            got.append([a[:19000] for a in s.state()])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
