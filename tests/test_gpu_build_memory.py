"""Stream-ordered scratch of the graph build at its peak, read from the device's
default memory pool: at most 70 bytes per point as the header says (24 more up to
2^21 points), with a last tree level that is nearly empty, nearly full or neither.
1 MiB is for what does not grow with the points."""
import ctypes

import pytest
import torch

import paper_2606_11402_gb300 as gg

pytestmark = pytest.mark.gpu
USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.mark.parametrize("N", [1 << 21, (1 << 21) + 1, 3_000_017, (1 << 22) - 1, (1 << 23) + 5])
@pytest.mark.parametrize("rule", [0, 1])
def test_build_scratch(N, rule):
    pts = torch.rand((N, 3), device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    pool, high = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    torch.cuda.synchronize()
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    gg.build_graph(pts, 4, split_rule=rule)
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert 0 < high.value <= (70 if N > 1 << 21 else 94) * N + (1 << 20)
