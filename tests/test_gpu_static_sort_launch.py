"""dem_sort_cells_static is made of ordinary launches: none asks for all its blocks to be
resident at once (a cooperative launch waits for a caller's kernel that holds SMs, and cannot
be captured into the body of a conditional graph node)."""
import ctypes

import pytest

from paper_1301_1714_gb300 import dem

pytestmark = pytest.mark.gpu

KERNEL_NODE = 0      # CU_GRAPH_NODE_TYPE_KERNEL
COOPERATIVE = 2      # CU_LAUNCH_ATTRIBUTE_COOPERATIVE


def test_no_cooperative_launch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1301_1714_gb300 import _build
    _build.build()
    cu = ctypes.CDLL("libcuda.so.1")
    dims, n = (64, 64, 32), 9001
    x = torch.rand((n, 3), dtype=torch.float64, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    out = torch.empty(n, **i32), torch.empty(n, **i32), torch.empty(64 * 64 * 32 + 1, **i32)
    s = torch.cuda.Stream()
    dem.dem_sort_cells_static(x, (0.0, 0.0, 0.0), 0.25, dims, *out, s.cuda_stream)   # first call outside a capture
    s.synchronize()
    stream, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(stream, 1) == 0                                # thread-local
    dem.dem_sort_cells_static(x, (0.0, 0.0, 0.0), 0.25, dims, *out, s.cuda_stream)
    assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    count = ctypes.c_size_t()
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    kernels = 0
    for node in nodes:
        kind, value = ctypes.c_int(), ctypes.create_string_buffer(64)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == KERNEL_NODE:
            kernels += 1
            assert cu.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), COOPERATIVE, value) == 0
            assert int.from_bytes(value.raw[:4], "little") == 0
    assert kernels > 0
    assert cu.cuGraphDestroy(graph) == 0
