"""Deep graphs whose level tables take a kernel just past the 48 KB of shared memory
that a launch gets by default: its dynamic part alone is below them, its static
part is not counted in.  The allocation-free NLL holds two words per level and
2 KB of static shared memory, so chains of 5884 to 6143 levels are between the two
limits; against graphgp_nll, whose sums differ in their FP64 order only (1e-9)."""
import numpy as np
import pytest
import torch

import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [5100, 5800, 5884, 6000, 6143, 6144, 8192])
def test_nll_noalloc_level_tables(L):
    g = gg.graph_import(workloads.uniform_cube(L, 81), 1, 1, np.arange(L, dtype=np.int32),
                        np.arange(L - 1, dtype=np.int32), np.arange(L + 1))
    assert g.num_levels == L
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, 0.1, 1e-6))
    v = to_gpu(workloads.white_noise(L, 82))
    want = gg.nll(g, f, v).item()
    out = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    gg.nll_noalloc(g, f, v, out)
    assert abs(out.item() - want) <= 1e-9 * abs(want)
