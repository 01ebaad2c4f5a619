"""The two-lanes-per-point factor (k <= 16) at the edges of its tiling: padded
rows (k not a multiple of 4), blocks of 64 points with 1, 63, 64 or 65 of
them, one more point than the resident grid, both forms of a row.  Against
the FP64 oracle within the stated 1e-4 (TOL), and the on-the-fly forms
against the stored factor bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, sigma_rel, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 8, 9, 12, 13, 15, 16])
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 700])
@pytest.mark.parametrize("kern", [(gg.MATERN12, 1.3, 0.2, 1e-3), (gg.MATERN32, 0.7, 0.15, 1e-3),
                                  (gg.MATERN52, 1.0, 0.1, 1e-2), (gg.SQEXP, 1.0, 0.08, 1e-2)])
def test_pair_factor_edges(k, rows, kern):
    n0 = 40
    pts = workloads.uniform_cube(n0 + rows, 7 * k + rows)
    g = gg.build_graph(to_gpu(pts), k, n0=n0)
    f = gg.factor(g, gg.Kernel(*kern))
    b, sigma, _ = f.export()
    w = oracle.build_graph(pts, k, n0=n0)
    fo = oracle.factor(w["pts_pos"], w["nbr_pos"], k, n0, oracle.Kernel(*kern))
    assert rel_norm(np_(b), fo["b"].reshape(rows, -1)[:, :k]) <= TOL
    assert sigma_rel(np_(sigma), fo["sigma"]) <= TOL
    xi = to_gpu(workloads.white_noise(n0 + rows, 1))
    v = gg.generate(g, f, xi)
    assert torch.equal(gg.generate_fused(g, gg.Kernel(*kern), xi), v)
    assert torch.equal(gg.whiten_fused(g, gg.Kernel(*kern), v), gg.whiten(g, f, v))
    vb, tb = gg.nll_backward(g, f, v)
    _, vf, tf = gg.nll_grad_fused(g, gg.Kernel(*kern), v)
    vo, to = oracle.nll_grad(w, oracle.Kernel(*kern), np_(v).astype(np.float64))
    for got_v, got_t in ((vb, tb), (vf, tf)):
        assert rel_norm(np_(got_v), vo) <= TOL
        assert np.abs(np_(got_t) - to).max() <= TOL * np.abs(to).max()


def test_pair_factor_grid_edge():
    """A last block of one point, beyond a whole number of resident grids."""
    n0, k = 256, 16
    grid = 3 * torch.cuda.get_device_properties(0).multi_processor_count * 64
    pts = torch.rand((n0 + 2 * grid + 1, 3), device="cuda")
    g = gg.build_graph(pts, k, n0=n0)
    kern = gg.Kernel(gg.MATERN32, 1.0, 0.1, 1e-6)
    f = gg.factor(g, kern)
    b, sigma, _ = f.export()
    order, nbr, _ = g.export()
    x = pts[order.long()].cpu().numpy()
    rows = np.r_[0, grid - 1, grid, 2 * grid - 1, 2 * grid]
    ko = oracle.Kernel(gg.MATERN32, 1.0, 0.1, 1e-6)
    got = np_(b)[rows]
    for r, row in zip(rows, got):
        c = np_(nbr)[r]
        K = np.array([[oracle.lib().oracle_kappa(1, 1.0, 0.1, float(np.linalg.norm(
            x[i].astype(np.float64) - x[j]))) for j in c] for i in c])
        kc = np.array([oracle.lib().oracle_kappa(1, 1.0, 0.1, float(np.linalg.norm(
            x[i].astype(np.float64) - x[n0 + r]))) for i in c])
        want = np.linalg.solve(K + ko.nugget * np.eye(k), kc)
        assert rel_norm(row, want) <= TOL * 10  # single rows: bound of the sampled-row checks
