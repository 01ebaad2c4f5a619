"""Waits under a tight max_spin.  The build's depths and the dense block of a factor
are computed by blocks that wait for each other, but their length is known, so no
setting of max_spin may end them: build, factor and what uses the dense block give
the results of the default setting bit for bit.  And every kind of wait runs out
when what it waits for never comes, is reported, and leaves the context usable."""
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


@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("spin", [1, 1000, 50_000])
def test_waits_run_out(which, spin):
    assert gg.selftest_wait(which, spin) == gg.ERR_TIMEOUT
    pts = to_gpu(workloads.uniform_cube(5000, 1))
    g = gg.build_graph(pts, 4, n0=50)
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, 0.1, 1e-6))
    xi = to_gpu(workloads.white_noise(5000, 2))
    back = gg.whiten(g, f, gg.generate(g, f, xi))
    assert gg.sync_status(g, f)[0] == 0
    assert torch.allclose(back, xi, rtol=1e-4, atol=1e-4)


def test_selftest_arguments():
    for which, spin in ((-1, 100), (3, 100), (1, 0), (2, (1 << 30) + 1)):
        assert gg.selftest_wait(which, spin) == gg.ERR_INVALID
