"""Waits under a tight max_spin.  The build's depths and the dense block of a factor
are computed by blocks that wait for each other, but their length is known, so no
setting of max_spin may end them: build, factor and what uses the dense block give
the results of the default setting bit for bit."""
import pytest
import torch

import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,k,n0", [(3000, 4, 0), (50_000, 16, 300), (20_000, 24, 700),
                                    (3000, 8, 2048)])
@pytest.mark.parametrize("rescue", [0.0, -1.0])
def test_tight_max_spin(N, k, n0, rescue):
    pts = to_gpu(workloads.uniform_cube(N, N))
    v = to_gpu(workloads.white_noise(N, 1))
    kern = gg.Kernel(gg.MATERN32, 1.0, 0.2, 1e-3, rescue)
    got = []
    for spin in (0, 1):
        g = gg.build_graph(pts, k, n0=n0, max_spin=spin)
        f = gg.factor(g, kern)
        assert gg.sync_status(g, f)[0] == 0
        gg.nll_grad_fused(g, kern, v)
        assert gg.sync_status(g, f)[0] == 0
        got.append((*g.export()[:2], *f.export(), gg.whiten(g, f, v),
                    gg.whiten_fused(g, kern, v)))
    for a, b in zip(*got):
        assert torch.equal(a, b)
