"""FP32 results to the last bit: digests of positions, velocities and spins after 30 steps on a
bed that keeps its contacts and springs, with neighbour lists and without, for few particles
and for many, recorded when every force pass ran one thread per particle (sm_103a, CUDA 13.0).
A pass that rounds any sum of products of the contact law differently changes them."""
import hashlib

import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu

LAWS = {"linear": {}, "hertz": dict(stiffness="hertz"), "simple": dict(model="simple"),
        "terms": dict(stiffness="hertz", terms=15, mu_roll=0.02, alpha_t=0.2, k_coh=2e3)}
RECORDED = {
    ("lists", 5003, "hertz"): "a1d36179dfb387a5",
    ("lists", 5003, "linear"): "a427961911af5a43",
    ("lists", 5003, "simple"): "ea4d8ff418136428",
    ("lists", 5003, "terms"): "bcb34989f708bde8",
    ("lists", 40003, "hertz"): "9fe725406f3e9818",
    ("lists", 40003, "linear"): "e2c2defcd624e4dd",
    ("lists", 40003, "simple"): "bd86120742a19068",
    ("lists", 40003, "terms"): "0da24c2acd5bfbb1",
    ("walk", 5003, "hertz"): "66caddde979fa862",
    ("walk", 5003, "linear"): "221ad8da2a0d0587",
    ("walk", 5003, "simple"): "a67d372187514b96",
    ("walk", 5003, "terms"): "114cdbb4cad16e83",
    ("walk", 21001, "hertz"): "b86cc0b425510ccb",
    ("walk", 21001, "linear"): "ae26546be48ed17a",
    ("walk", 21001, "simple"): "5c1319bb99eb7a48",
    ("walk", 21001, "terms"): "4fddc3f596e1050d",
}


def digest(policy, n, law):
    sc = scenes.drum(seed=11, n=n, precision="fp32")
    x = sc.x * 0.998
    v = sc.v + scenes.uniform(12, 3 * n, -0.1, 0.1).reshape(n, 3)
    w = sc.w + scenes.uniform(13, 3 * n, -5.0, 5.0).reshape(n, 3)
    p = sc.params.copy(**LAWS[law])
    if policy == "lists":
        p = p.copy(resort_interval=0, skin=1e-4, cell_size=p.cell_size + 1e-4)
    with dem.Simulation(p, x, v, w, sc.r) as s:
        s.step(30)
        out = s.state()
    return hashlib.sha256(b"".join(np.ascontiguousarray(a).tobytes() for a in out)).hexdigest()[:16]


@pytest.mark.parametrize("law", sorted(LAWS))
@pytest.mark.parametrize("policy,n", [("lists", 5003), ("lists", 40003), ("walk", 5003), ("walk", 21001)])
def test_same_bits_as_recorded(policy, n, law):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    assert digest(policy, n, law) == RECORDED[policy, n, law]
