"""dem_sort_cells_static at the edges of its work split (blocks, scan tiles), against numpy,
and replayed from a captured graph."""
import numpy as np
import pytest

from paper_1301_1714_gb300 import dem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    dem.lib()
    return torch


def _reference(x, cell, dims):
    c = np.clip(np.floor(x / cell), 0, np.array(dims) - 1).astype(np.int64) if len(x) else np.zeros((0, 3), np.int64)
    key = (c[:, 2] * dims[1] + c[:, 1]) * dims[0] + c[:, 0]
    start = np.searchsorted(np.sort(key), np.arange(dims[0] * dims[1] * dims[2] + 1))
    return key, np.argsort(key, kind="stable"), start


def _buffers(torch, n, dims):
    i32 = dict(dtype=torch.int32, device="cuda")
    return torch.full((n,), -1, **i32), torch.full((n,), -1, **i32), torch.full((dims[0] * dims[1] * dims[2] + 1,), -1, **i32)


@pytest.mark.parametrize("n", [0, 1, 255, 257, 4096, 77823, 77825, 155649, 262144])
@pytest.mark.parametrize("dims", [(1, 2, 1), (23, 89, 1), (128, 16, 1), (61, 67, 73), (128, 128, 64)])
def test_sizes(torch, n, dims):
    if n > 100 * dims[0] * dims[1] * dims[2]:
        pytest.skip("quadratic in the cells' occupancy")
    rng = np.random.default_rng(n + dims[0])
    x = rng.uniform(-0.5, np.array(dims) + 0.5, size=(n, 3)) * 0.25
    xd = torch.tensor(x, device="cuda")
    out = _buffers(torch, n, dims)
    for _ in range(2):
        dem.dem_sort_cells_static(xd, (0.0, 0.0, 0.0), 0.25, dims, *out)
        torch.cuda.synchronize()
        for got, want in zip(out, _reference(x, 0.25, dims)):
            assert np.array_equal(got.cpu().numpy(), want)


def test_captured_in_a_graph(torch):
    dims, n = (31, 17, 19), 9001
    xd = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    out = _buffers(torch, n, dims)
    s = torch.cuda.Stream()
    dem.dem_sort_cells_static(xd, (0.0, 0.0, 0.0), 0.25, dims, *out, s.cuda_stream)   # first call outside a capture
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        dem.dem_sort_cells_static(xd, (0.0, 0.0, 0.0), 0.25, dims, *out, s.cuda_stream)
    for seed in (1, 2):
        x = np.random.default_rng(seed).uniform(0, 1, size=(n, 3)) * np.array(dims) * 0.25
        xd.copy_(torch.tensor(x))
        g.replay()
        torch.cuda.synchronize()
        for got, want in zip(out, _reference(x, 0.25, dims)):
            assert np.array_equal(got.cpu().numpy(), want)
