"""A step that overflows a particle's contact slots while another error is reported first (a
particle that leaves the finite range, a full neighbour list): the overflow's void step is not
left standing, which would make every later step do nothing and succeed."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lists,slots", [(False, 64), (True, 4)])
@pytest.mark.parametrize("own_stream", [False, True])
def test_later_steps_run_or_report(lists, slots, own_stream):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    stream = torch.cuda.Stream().cuda_stream if own_stream else None
    p = scenes.drum(seed=1, n=500, precision="fp32").params.copy(walls=[])
    if lists:
        p = p.copy(resort_interval=0, skin=1e-4, cell_size=p.cell_size + 1e-4)
    n = 140
    x, v = 1e-4 * scenes.uniform(3, 3 * n, -1.0, 1.0).reshape(n, 3), np.zeros((n, 3))   # a cluster: all overlap
    if not lists:
        x[:40, 0], v[:40, 0] = 3.40282e38, 3.4e38          # 40 runaways; 100 spheres of 99 contacts
    with dem.Simulation(p, x, v, np.zeros((n, 3)), np.full(n, 1e-3, np.float32), cuda_stream=stream,
                        max_contacts=slots) as s:
        with pytest.raises(dem.DemError) as e:
            s.step(4)
        assert e.value.status in (dem.DEM_ERR_NONFINITE, dem.DEM_ERR_CAPACITY)
        for k in (1, 3):
            before = s.state()[0][-1].copy()
            try:
                s.step(k)
            except dem.DemError as err:
                assert err.status in (dem.DEM_ERR_NONFINITE, dem.DEM_ERR_CAPACITY)
            else:
                assert not np.array_equal(before, s.state()[0][-1])
