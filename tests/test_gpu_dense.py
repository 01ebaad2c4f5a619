"""The dense initial block at the edges of its tiling: sizes around the 32 x 32
tiles, the switch of the summation order (n0 = 320), the switch of the inverse's
rows per warp (288) and more tile rows than a side of the block grid (n0 > 384),
in FP32 and (rescue_tol < 0, or an ill-conditioned block) in FP64, against
torch in FP64 on the same coordinates.  L0 within the stated 1e-4 norm-wise,
the inverse through xi_0 = L0^-1 v_0."""
import math

import pytest
import torch

import paper_2606_11402_gb300 as gg
from gpu_util import TOL

pytestmark = pytest.mark.gpu


def kappa32(x, ell):
    a = math.sqrt(3.0) * torch.cdist(x, x, compute_mode="donot_use_mm_for_euclid_dist") / ell
    return (1.0 + a) * torch.exp(-a)


@pytest.mark.parametrize("n0", [1, 2, 31, 32, 33, 64, 95, 255, 256, 257, 288, 289, 320, 321, 385,
                                1000, 2048])
@pytest.mark.parametrize("ell,nugget,rescue", [(0.05, 1e-2, 0.0), (0.05, 1e-2, -1.0),
                                               (1.0, 1e-5, 0.0)])
def test_dense_block_edges(n0, ell, nugget, rescue):
    gen = torch.Generator(device="cuda").manual_seed(n0)
    pts = torch.rand((n0 + 3, 3), generator=gen, device="cuda")
    g = gg.build_graph(pts, 1, n0=n0)
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, ell, nugget, rescue))
    _, sigma, L0 = f.export()
    order, _, _ = g.export()
    x = pts[order.long()][:n0].double()
    K = kappa32(x, ell) + nugget * torch.eye(n0, dtype=torch.float64, device="cuda")
    want = torch.linalg.cholesky(K)
    assert torch.equal(L0, torch.tril(L0))
    assert torch.equal(sigma[:n0], L0.diagonal())
    assert (L0 - want).norm() <= TOL * want.norm()
    assert (sigma[:n0].double() / want.diagonal() - 1).abs().max() <= TOL
    v = torch.randn(n0 + 3, generator=gen, device="cuda")
    v[:n0] = (want @ torch.randn(n0, generator=gen, device="cuda").double()).float()
    xi0 = torch.linalg.solve_triangular(want, v[:n0, None].double(), upper=False)[:, 0]
    got = gg.whiten(g, f, v)[:n0].double()
    # v_0 is rounded to FP32: a relative 2^-24 per entry through L0^-1
    amp = torch.linalg.matrix_norm(torch.linalg.inv(want), 2) * v[:n0].norm() / xi0.norm()
    assert (got - xi0).norm() <= (TOL + 2.0 ** -22 * amp) * xi0.norm()
    status, bad = gg.sync_status(g, f)
    assert status == gg.OK and bad == 0
