"""The root and reciprocal of the FP32 factors, and the factors where their
arguments leave the normal range.

One Newton step on an estimate of relative error 2^-22.4 leaves 2^-44, which is
2^-20 ulp: an argument is rounded wrongly, by one ulp, only if its root lies that
close to a rounding boundary, 2^-19 of the arguments on average.  For the
reciprocal (estimate 2^-23, exact residual) it is 2^-21.  Twice that many are
allowed.  References are FP64 results rounded to FP32, correctly rounded as 53 >=
2 24 + 2."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import TOL, np_, rel_norm, sigma_rel, to_gpu

pytestmark = pytest.mark.gpu


def run(x):
    return [np_(t) for t in gg.selftest_roots(to_gpu(x))]


def ulps(got, want):
    return np.abs(got.view(np.int32).astype(np.int64) - want.view(np.int32))


def test_every_mantissa():
    x = np.arange(0x3f800000, 0x40800000, dtype=np.int32).view(np.float32)  # [1, 4)
    root, pair, inv = run(x)
    d = ulps(root, np.sqrt(x.astype(np.float64)).astype(np.float32))
    assert d.max() <= 1 and (d > 0).sum() <= 2 * len(x) * 2.0**-19
    assert np.array_equal(root, pair)
    d = ulps(inv, (1.0 / x.astype(np.float64)).astype(np.float32))
    assert d.max() <= 1 and (d > 0).sum() <= 2 * len(x) * 2.0**-21


def test_every_exponent():
    rng = np.random.default_rng(7)
    bits = [[0, 0x00800000, 0x00800001, 0x7f7fffff]]
    bits += [rng.integers(e << 23, (e + 1) << 23, 1 << 14) for e in range(1, 255)]
    x = np.concatenate(bits).astype(np.int32).view(np.float32)
    x = x[rng.permutation(len(x))]
    root, pair, inv = run(x)
    want = np.sqrt(x.astype(np.float64)).astype(np.float32)
    assert ulps(root, want).max() <= 1
    assert np.array_equal(root[x == 0], x[x == 0])
    assert np.array_equal(root, pair)
    ok = (x > 0) & (x <= 2.0**126)
    assert ulps(inv[ok], (1.0 / x[ok].astype(np.float64)).astype(np.float32)).max() <= 1
    root, pair, _ = run(np.array([np.inf, 1.0, 2.0, np.inf], np.float32))
    assert np.array_equal(np.isnan(root), [1, 0, 0, 1]) and np.array_equal(np.isnan(pair), [1, 0, 0, 1])


@pytest.mark.parametrize("kern", [gg.MATERN12, gg.MATERN32, gg.MATERN52])
@pytest.mark.parametrize("k", [8, 24, 48])
@pytest.mark.parametrize("scale,sigma2,nugget", [(2.0**-58, 1.0, 1e-2), (1.0, 2.0**-125, 0.2)])
def test_factor_below_the_normal_range(kern, k, scale, sigma2, nugget):
    """Squared distances, or pivots, that are subnormal (these keep 20 bits and more):
    the factor is within the stated 1e-4 of the FP64 one, also of an imported graph."""
    n0, N = 64, 500
    pts = (workloads.uniform_cube(N, 11) * np.float32(scale)).astype(np.float32)
    g = gg.build_graph(to_gpu(pts), k, n0=n0)
    args = (kern, sigma2, 0.3 * scale, nugget * sigma2)
    f = gg.factor(g, gg.Kernel(*args))
    assert gg.sync_status(g, f)[0] == 0
    order, nbr, lo = g.export()
    fi = gg.factor(gg.graph_import(pts, k, n0, np_(order), np_(nbr), lo.numpy()), gg.Kernel(*args))
    assert all(torch.equal(a, c) for a, c in zip(f.export(), fi.export()))
    fo = oracle.factor(pts[np_(order)], np_(nbr).reshape(N - n0, k), k, n0, oracle.Kernel(*args))
    b, sigma, L0 = (np_(t) for t in f.export())
    assert rel_norm(b, fo["b"].reshape(N - n0, -1)[:, :k]) <= TOL
    assert sigma_rel(sigma, fo["sigma"]) <= TOL
    if k <= 32:  # the on-the-fly form decides the same
        xi = to_gpu(workloads.white_noise(N, 3))
        assert torch.equal(gg.generate_fused(g, gg.Kernel(*args), xi), gg.generate(g, f, xi))


@pytest.mark.parametrize("kern", [gg.MATERN12, gg.MATERN32, gg.MATERN52, gg.SQEXP])
@pytest.mark.parametrize("k", [8, 24, 48])
@pytest.mark.parametrize("e", [-58, -100])
def test_cloud_scaled_by_a_power_of_two(kern, k, e):
    """The same graph on points and lengthscale scaled down until squared distances
    vanish in FP32: the factor is the same bit for bit, and the gradients are, in the
    scaled unit, up to the order of their sums (1e-5 of the largest)."""
    n0, N = 70, 600
    pts = workloads.uniform_cube(N, 12)
    g = gg.build_graph(to_gpu(pts), k, n0=n0)
    order, nbr, lo = g.export()
    v = to_gpu(workloads.white_noise(N, 5))
    got = []
    for s in (1.0, 2.0**e):
        gi = gg.graph_import((pts * np.float32(s)).astype(np.float32), k, n0, np_(order), np_(nbr),
                             lo.numpy())
        kn = gg.Kernel(kern, 1.0, 0.2 * s, 1e-2)
        f = gg.factor(gi, kn)
        vb, tb = gg.nll_backward(gi, f, v)
        pb = gg.nll_backward_points(gi, f, v)
        fused = gg.nll_grad_fused(gi, kn, v)[1:] if k <= 32 else (vb, tb)
        unit = torch.tensor([s, 1.0, 1.0], device="cuda", dtype=torch.float64)
        got.append((f.export(), gg.nll(gi, f, v).item(),
                    [vb, tb * unit, pb.double() * s, fused[0], fused[1] * unit]))
    for a, b in zip(got[0][0], got[1][0]):
        assert torch.equal(a, b)
    assert abs(got[0][1] - got[1][1]) <= 1e-12 * abs(got[0][1])
    for a, b in zip(got[0][2], got[1][2]):
        assert (a - b).abs().max() <= 1e-5 * a.abs().max()
