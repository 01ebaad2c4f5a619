"""The eight-lanes-per-point factor (16 < k <= 32) at the edges of its tiling:
both padded sizes (24 and 32) and all row lengths, blocks of 16 points with 1,
15, 16 or 17 of them, both forms of a row; FP64 rescue of every row.  Against
the FP64 oracle within the stated 1e-4 (TOL), and the on-the-fly forms against
the stored factor bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, sigma_rel, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [17, 19, 20, 21, 24, 25, 28, 29, 31, 32])
@pytest.mark.parametrize("rows", [1, 15, 16, 17, 300])
@pytest.mark.parametrize("kern", [(gg.MATERN12, 1.3, 0.2, 1e-3), (gg.MATERN32, 0.7, 0.15, 1e-3),
                                  (gg.MATERN52, 1.0, 0.1, 1e-2), (gg.SQEXP, 1.0, 0.08, 1e-2)])
@pytest.mark.parametrize("rescue", [0.0, -1.0])
def test_oct_factor_edges(k, rows, kern, rescue):
    n0 = 40
    pts = workloads.uniform_cube(n0 + rows, 7 * k + rows)
    kn = gg.Kernel(*kern, rescue)
    g = gg.build_graph(to_gpu(pts), k, n0=n0)
    f = gg.factor(g, kn)
    b, sigma, _ = f.export()
    w = oracle.build_graph(pts, k, n0=n0)
    fo = oracle.factor(w["pts_pos"], w["nbr_pos"], k, n0, oracle.Kernel(*kern))
    assert rel_norm(np_(b), fo["b"].reshape(rows, -1)[:, :k]) <= TOL
    assert sigma_rel(np_(sigma), fo["sigma"]) <= TOL
    xi = to_gpu(workloads.white_noise(n0 + rows, 1))
    v = gg.generate(g, f, xi)
    assert torch.equal(gg.generate_fused(g, kn, xi), v)
    assert torch.equal(gg.whiten_fused(g, kn, v), gg.whiten(g, f, v))
    vb, tb = gg.nll_backward(g, f, v)
    _, vf, tf = gg.nll_grad_fused(g, kn, v)
    vo, to = oracle.nll_grad(w, oracle.Kernel(*kern), np_(v).astype(np.float64))
    for got_v, got_t in ((vb, tb), (vf, tf)):
        assert rel_norm(np_(got_v), vo) <= TOL
        assert np.abs(np_(got_t) - to).max() <= TOL * np.abs(to).max()
