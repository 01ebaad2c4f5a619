"""generate, whiten and generate_backward where a deep graph takes the sweeps from
one kernel to the next by its number of levels: the one-block runs end at 4096, the
sweep without barriers takes no more than 4096, the tiled whiten 8192.  Layers of w
points, each conditioned on two points of the layer before; against the exported
rows applied level by level in FP64, within the stated 1e-4 (TOL)."""
import numpy as np
import pytest

import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4095, 4096, 4097, 4098, 9000])
@pytest.mark.parametrize("w,k", [(2, 2), (7, 2), (23, 2), (30, 20)])
def test_layers(L, w, k):
    N, n0 = L * w, w
    p = np.arange(n0, N)
    nbr = (p // w - 1)[:, None] * w + (p[:, None] + np.arange(k)) % w
    pts = np.cumsum(workloads.uniform_cube(N, L + w), axis=0, dtype=np.float64) / w
    g = gg.graph_import((pts % 8).astype(np.float32), k, n0, np.arange(N), nbr.astype(np.int32),
                        np.arange(0, N + 1, w))
    assert g.num_levels == L
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, 1.0, 1e-2))
    xi, vbar = (to_gpu(workloads.white_noise(N, s)) for s in (3, 4))
    v = gg.generate(g, f, xi)
    x = gg.whiten(g, f, v)
    xb, _ = gg.generate_backward(g, f, xi, v, vbar, theta=False)
    assert gg.sync_status(g, f)[0] == 0
    b, sigma, L0 = (np_(t).astype(np.float64) for t in f.export())
    b, xe, ve = b.reshape(N - n0, k), np_(xi).astype(np.float64), np.zeros(N)
    ve[:n0] = np.tril(L0) @ xe[:n0]
    for s in range(n0, N, w):
        ve[s:s + w] = (b[s - n0:s - n0 + w] * ve[nbr[s - n0:s - n0 + w]]).sum(1) + \
            sigma[s:s + w] * xe[s:s + w]
    assert rel_norm(np_(v), ve) <= TOL
    assert rel_norm(np_(x), xe) <= TOL
    u = np_(vbar).astype(np.float64)
    for s in range(N - w, n0 - 1, -w):
        np.add.at(u, nbr[s - n0:s - n0 + w], b[s - n0:s - n0 + w] * u[s:s + w, None])
    want = sigma * u
    want[:n0] = np.tril(L0).T @ u[:n0]
    assert rel_norm(np_(xb), want) <= TOL
