"""The dense part of the backward at the edges of its tiles (32 columns, 256 rows
a chunk, 32 x 32 of a product), against the oracle and the exported block; the
generate VJP where the run of small levels ends (4096 row entries a level),
against the exported rows applied level by level in FP64.  Within the stated
1e-4 (TOL)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0", [1, 31, 32, 33, 64, 255, 256, 257, 289, 700])
def test_dense_backward_edges(n0):
    N, kern = n0 + 3, (gg.MATERN32, 1.0, 0.1, 1e-2)
    pts = workloads.uniform_cube(N, n0)
    g = gg.build_graph(to_gpu(pts), 1, n0=n0)
    kn = gg.Kernel(*kern)
    f = gg.factor(g, kn)
    xi = to_gpu(workloads.white_noise(N, 1))
    v = gg.generate(g, f, xi)
    w = oracle.build_graph(pts, 1, n0=n0)
    vo, to = oracle.nll_grad(w, oracle.Kernel(*kern), np_(v).astype(np.float64))
    vb, tb = gg.nll_backward(g, f, v)
    assert rel_norm(np_(vb), vo) <= TOL
    assert np.abs(np_(tb) - to).max() <= TOL * np.abs(to).max()
    part, tp = (torch.zeros(s, device="cuda", dtype=d) for s, d in ((N, torch.float32),
                                                                   (3, torch.float64)))
    for p in ((0, n0), (n0, N)):  # the row-range form adds the dense part to the sparse one
        fr = gg.factor_rows(g, kn, *p)
        gg.nll_backward_rows(g, fr, v, part, thetabar=tp)
    assert rel_norm(np_(part), vo) <= TOL
    assert np.abs(np_(tp) - to).max() <= TOL * np.abs(to).max()
    vbar = torch.zeros(N, device="cuda")
    vbar[:n0] = xi[:n0] + 1.0
    xb, _ = gg.generate_backward(g, f, xi, v, vbar, theta=False)
    L0 = np_(f.export()[2]).astype(np.float64)
    assert rel_norm(np_(xb)[:n0], L0.T @ np_(vbar)[:n0].astype(np.float64)) <= TOL


@pytest.mark.parametrize("k", [4, 7, 12, 16, 20, 28, 32, 48, 64])
@pytest.mark.parametrize("N", [101, 150, 2000, 5003, 40000])
def test_generate_vjp_levels(N, k):
    n0 = 100
    g = gg.build_graph(to_gpu(workloads.uniform_cube(N, N + k)), k, n0=n0)
    f = gg.factor(g, gg.Kernel(gg.MATERN32, 1.0, 0.2, 1e-3))
    xi, vbar = (to_gpu(workloads.white_noise(N, s)) for s in (3, 4))
    v = gg.generate(g, f, xi)
    xb, _ = gg.generate_backward(g, f, xi, v, vbar, theta=False)
    assert gg.sync_status(g, f)[0] == 0
    _, nbr, lo = g.export()
    nbr, lo = np_(nbr).reshape(N - n0, k).astype(np.int64), lo.numpy()
    b, sigma, L0 = (np_(t).astype(np.float64) for t in f.export())
    b = b.reshape(N - n0, k)
    u = np_(vbar).astype(np.float64)
    for s, e in list(zip(lo[1:-1], lo[2:]))[::-1]:
        np.add.at(u, nbr[s - n0:e - n0], b[s - n0:e - n0] * u[s:e, None])
    want = sigma * u
    want[:n0] = L0.T @ u[:n0]
    assert rel_norm(np_(xb), want) <= TOL
