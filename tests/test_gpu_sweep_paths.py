"""generate and whiten where the way through the levels changes: clouds that one
block finishes (every level up to 1024 points), clouds whose first large level
ends that block's run, row entries just below and above the line of the
barrier-free sweep, tiles just below and above four per SM; all lane splits.
Against the exported rows applied level by level in FP64: an entry is a sum of at
most k + 1 products in FP32.  whiten is within (k + 4) 2^-24 of the sum of absolute
values, entry by entry; generate carries such errors through the levels, and is
within the stated 1e-4 (TOL)."""
import numpy as np
import pytest
import torch

import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, to_gpu

pytestmark = pytest.mark.gpu


def check(pts, k, n0):
    N = len(pts)
    g = gg.build_graph(to_gpu(pts), k, n0=n0)
    kn = gg.Kernel(gg.MATERN32, 1.0, 0.2, 1e-3)
    f = gg.factor(g, kn)
    xi = to_gpu(workloads.white_noise(N, 3))
    v = gg.generate(g, f, xi)
    x = gg.whiten(g, f, v)
    assert gg.sync_status(g, f)[0] == 0
    n0 = g.n0
    nbr, lo = (np_(t) for t in g.export()[1:3])
    b, sigma, L0 = (np_(t).astype(np.float64) for t in f.export())
    nbr, b = nbr.reshape(N - n0, -1)[:, :k].astype(np.int64), b.reshape(N - n0, -1)[:, :k]
    xe, ve = np_(xi).astype(np.float64), np.zeros(N)
    ve[:n0] = np.tril(L0.reshape(n0, n0)) @ xe[:n0]
    for s, e in zip(lo[1:-1], lo[2:]):
        ve[s:e] = (b[s - n0:e - n0] * ve[nbr[s - n0:e - n0]]).sum(1) + sigma[s:e] * xe[s:e]
    assert rel_norm(np_(v), ve) <= TOL
    v64 = np_(v).astype(np.float64)
    res = v64[n0:] - (b * v64[nbr]).sum(1)
    scale = (np.abs(b) * np.abs(v64[nbr])).sum(1) + np.abs(v64[n0:])
    err = np.abs(np_(x)[n0:] * sigma[n0:] - res)
    assert (err <= (k + 4) * 2.0**-24 * scale).all()


@pytest.mark.parametrize("k", [4, 7, 12, 16, 20, 32, 48, 64])
@pytest.mark.parametrize("N", [200, 3001, 40000])
def test_small_and_medium(N, k):
    check(workloads.uniform_cube(N, N + k), k, 100)


@pytest.mark.parametrize("k", [16, 20, 32, 48, 64])
@pytest.mark.parametrize("side", [0, 1])
def test_entries_line(k, side):
    check(workloads.uniform_cube((8 << 20) // k + side, k), k, 100)


@pytest.mark.parametrize("side", [-1, 1])
def test_tiles_line(side):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check(workloads.uniform_cube(4096 * (4 * sms - (side < 0)), 5), 4, 100)


def test_nan_in_one_entry_spreads_and_ends():
    """A NaN with all bits set in xi is the not-yet mark of the barrier-free sweep:
    the result is NaN, not a wait."""
    N, k = 60000, 16
    g = gg.build_graph(to_gpu(workloads.uniform_cube(N, 9)), k)
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, 0.2, 1e-3))
    xi = to_gpu(workloads.white_noise(N, 3))
    for pos in (0, g.n0 + 1, N // 2, N - 1):
        x = xi.clone()
        x.view(torch.int32)[pos] = -1
        v = gg.generate(g, f, x)
        assert gg.sync_status(g, f)[0] == 0
        assert torch.isnan(v[pos]) and not torch.isnan(v[:min(pos, g.n0)]).any()
