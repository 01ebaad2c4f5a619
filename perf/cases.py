"""Cases for timing the library: what programs built on it have it do.

A case names a path through the public entry points and the sizes and options
of one problem.  The paths:

  build     build_graph and the arrays it gives (once per point cloud)
  factor    factor for a kernel, its arrays and log-determinant
  sweep     generate, whiten of the result, logdet with a stored factor
  vjp       generate and its VJP with a stored factor (a field fitted to data
            under a fixed kernel)
  fit       autograd.nll_fit forward and backward (kernel parameters that
            change at every step: no factor is stored)
  gradient  autograd.nll forward and backward (factor, NLL, adjoints); with
            ``points`` also the gradient of the coordinates
  fly       generate_fused and nll_fused: Alg. 1 as printed

Kernel parameters under an optimiser are float32 logarithms, as a parameter
of a torch module is.  Fields that are given (the data) are realisations of
the kernel's process by random Fourier features, plus nugget noise.
``exact`` builds the graph, the conditionals, the sweeps and the gradients
again in plain torch, in 64 bits (the neighbour keys in the 32-bit arithmetic
that defines them).
"""
from __future__ import annotations

import math

import torch

import paper_2606_11402_gb300 as gg
from paper_2606_11402_gb300 import autograd as ag

# Largest problem that exact() works out, by brute force over all pairs.
EXACT_MAX = 1 << 18


def _case(name, path, cloud, N, k, kernel, ell, nugget, d=3, n0=0, rescue=0.0, points=False):
    return dict(name=name, path=path, cloud=cloud, N=N, d=d, k=k, n0=n0, kernel=kernel, ell=ell,
                nugget=nugget, rescue=rescue, points=points)


def listed():
    return [
        # the tiny workload: launches and level latency are all there is
        _case("sweep_tiny", "sweep", "uniform", 4096, 8, gg.MATERN32, 0.1, 1e-6),
        # a served instance of mean size, clustered (its cloud has 100 blobs)
        _case("sweep_served", "sweep", "blobs100", 127_001, 16, gg.MATERN32, 0.05, 1e-6),
        # the headline workload: 2^26 unit-Gaussian points
        _case("sweep_headline", "sweep", "gaussian", 1 << 26, 16, gg.MATERN32, 0.1, 1e-6),
        # a small planar cloud: graph of a map or an image
        _case("build_planar", "build", "uniform", 30_011, 8, gg.MATERN32, 0.1, 1e-6, d=2),
        # the scale workload's clustered cloud at the size of a large survey
        _case("build_clustered", "build", "blobs10000", 1 << 24, 16, gg.MATERN32, 0.02, 1e-6),
        # a factor of the headline cloud, kept for many sweeps
        _case("factor_headline", "factor", "gaussian", 1 << 24, 16, gg.MATERN32, 0.1, 1e-6),
        # the large-dynamic-range workload: no nugget, many rows need FP64
        _case("factor_range", "factor", "ldr", 1 << 20, 16, gg.MATERN32, 0.05, 0.0,
              rescue=2.0 ** -10),
        # a fit step on a small data set, odd sizes
        _case("fit_small", "fit", "uniform", 10_007, 10, gg.MATERN52, 0.15, 1e-3),
        # a fit step on a large cloud
        _case("fit_large", "fit", "gaussian", 1 << 22, 16, gg.MATERN32, 0.1, 1e-6),
        # the differentiation workload (squared exponential, k = 32)
        _case("gradient_k32", "gradient", "uniform", 1 << 20, 32, gg.SQEXP, 0.03, 1e-4),
        # inference of a field of a million points, the kernel fixed
        _case("vjp_million", "vjp", "gaussian", 1_000_003, 16, gg.MATERN32, 0.1, 1e-6),
        # the paper's benchmark form: unit Gaussian, n0 = 1000, nothing stored
        _case("fly_paper", "fly", "gaussian", 1 << 20, 16, gg.MATERN32, 0.1, 1e-6, n0=1000),
    ]


def draw(rng):
    # largest N by path (gradient: at k = 32; N k^2 is kept below that)
    top = dict(build=1 << 23, factor=1 << 23, sweep=1 << 24, vjp=1 << 20, fit=1 << 21,
               gradient=1 << 19, fly=1 << 20)
    path = rng.choice(sorted(top))
    ks = [4, 7, 8, 12, 13, 16, 16, 20, 24, 32] + ([48, 64] if path not in ("fit", "fly") else [])
    k = rng.choice(ks)
    most = top[path] * min(1.0, (24.0 / k) ** 2)
    N = int(round(math.exp(rng.uniform(math.log(2000), math.log(most)))))
    kernel = rng.choice([gg.MATERN12, gg.MATERN32, gg.MATERN32, gg.MATERN52, gg.SQEXP])
    d = rng.choice([1, 2, 3, 3, 3])
    cloud = rng.choice(["uniform", "gaussian", "blobs100"] if d == 3 else ["uniform", "gaussian"])
    # lengthscales of a few mean spacings (smooth kernels: nearer to the
    # spacing, with a nugget that bounds the conditioning)
    spacing = N ** (-1.0 / d)
    smooth = kernel in (gg.MATERN52, gg.SQEXP)
    ell = min(0.2, spacing * rng.uniform(3.0, 6.0 if smooth else 20.0))
    nugget = rng.choice([1e-3, 1e-2] if smooth else [1e-6, 1e-4, 1e-2])
    n0 = rng.choice([0, 0, 0, 64, 300, 1000])
    return dict(path=path, cloud=cloud, N=N, d=d, k=k, n0=n0 if k <= n0 <= N else 0, kernel=kernel,
                ell=ell, nugget=nugget, rescue=0.0,
                points=path == "gradient" and rng.random() < 0.3)


# ---- inputs -----------------------------------------------------------------
def _cloud(case, gen):
    N, d, kind = case["N"], case["d"], case["cloud"]
    dev = torch.device("cuda")
    if kind == "uniform":
        return torch.rand((N, d), generator=gen, device=dev)
    if kind == "gaussian":
        return torch.randn((N, d), generator=gen, device=dev)
    if kind == "ldr":  # 90 % radii log-uniform in [1e-3, 1], 10 % uniform in [-1, 1]^3
        x = torch.randn((N, d), generator=gen, device=dev)
        x /= x.norm(dim=1, keepdim=True)
        x *= 10.0 ** (-3.0 * torch.rand((N, 1), generator=gen, device=dev))
        back = torch.rand(N, generator=gen, device=dev) < 0.1
        uni = 2.0 * torch.rand((N, d), generator=gen, device=dev) - 1.0
        return torch.where(back[:, None], uni, x).contiguous()
    # Gaussian blobs of log-uniform width in [1e-4, 1e-1], 10 % uniform background
    n = int(kind[5:])
    centres = torch.rand((n, d), generator=gen, device=dev)
    widths = 10.0 ** (-4.0 + 3.0 * torch.rand((n, 1), generator=gen, device=dev))
    which = torch.randint(0, n, (N,), generator=gen, device=dev)
    x = centres[which] + widths[which] * torch.randn((N, d), generator=gen, device=dev)
    back = torch.rand(N, generator=gen, device=dev) < 0.1
    uni = torch.rand((N, d), generator=gen, device=dev)
    return torch.where(back[:, None], uni, x).contiguous()


def _field(case, pts, gen):
    """A realisation of the process at the points (input order): 64 random
    Fourier features of the kernel's spectral density, and nugget noise."""
    dev, F = pts.device, 64
    dof = {gg.MATERN12: 1, gg.MATERN32: 3, gg.MATERN52: 5}.get(case["kernel"])
    w = torch.randn((F, case["d"]), generator=gen, device=dev) / case["ell"]
    if dof:
        chi = torch.randn((F, dof), generator=gen, device=dev).square().sum(1, keepdim=True)
        w = w * torch.sqrt(dof / chi)
    phase = 2.0 * math.pi * torch.rand(F, generator=gen, device=dev)
    out = math.sqrt(case["nugget"]) * torch.randn(len(pts), generator=gen, device=dev)
    for f in range(F):
        t = torch.zeros_like(out)
        for c in range(case["d"]):
            t += pts[:, c] * w[f, c]
        out += math.sqrt(2.0 / F) * torch.cos(t + phase[f])
    return out


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    pts = _cloud(case, gen)
    path, s = case["path"], dict(points=pts)
    if path in ("sweep", "vjp", "fly"):
        s["xi"] = torch.randn(case["N"], generator=gen, device="cuda")
    if path in ("vjp", "fit", "gradient", "fly"):
        s["field"] = _field(case, pts, gen)
    if path in ("fit", "gradient"):
        theta = torch.tensor([case["ell"], 1.0, case["nugget"]], dtype=torch.float64).log()
        s["log_theta"] = theta.float()
    return s


def _kernel(case):
    return gg.Kernel(case["kernel"], 1.0, case["ell"], case["nugget"], case["rescue"])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], s["kern"] = case, _kernel(case)
    if case["path"] == "build":
        return s
    s["graph"] = gg.build_graph(s["points"], case["k"], n0=case["n0"])
    if "field" in s:  # the data, in graph order
        order, _, _ = s["graph"].export()
        s["field"] = s["field"][order.long()].contiguous()
    if case["path"] in ("sweep", "vjp"):
        s["factor"] = gg.factor(s["graph"], s["kern"])
    return s


def run(s):
    case, path, g = s["case"], s["case"]["path"], s.get("graph")
    if path == "build":
        g = gg.build_graph(s["points"], case["k"], n0=case["n0"])
        order, nbr, _ = g.export()
        _, _, _, depth, _ = g.export_tree()
        return dict(order=order, nbr=nbr, depth=depth)
    if path == "factor":
        f = gg.factor(g, s["kern"])
        b, sigma, L0 = f.export()
        return dict(b=b, sigma=sigma, L0=L0, logdet=gg.logdet(f))
    if path == "sweep":
        v = gg.generate(g, s["factor"], s["xi"])
        return dict(v=v, xi=gg.whiten(g, s["factor"], v), logdet=gg.logdet(s["factor"]))
    if path == "vjp":
        v = gg.generate(g, s["factor"], s["xi"])
        xibar, _ = gg.generate_backward(g, s["factor"], s["xi"], v, v - s["field"], theta=False)
        return dict(v=v, xibar=xibar)
    if path == "fly":
        v = gg.generate_fused(g, s["kern"], s["xi"])
        return dict(v=v, nll=gg.nll_fused(g, s["kern"], s["field"]))
    v = s["field"].detach().requires_grad_(True)
    log_theta = s["log_theta"].detach().requires_grad_(True)
    theta = log_theta.double().exp()
    if path == "fit":
        loss = ag.nll_fit(g, case["kernel"], theta, v)
        loss.backward()
        return dict(nll=loss.detach(), v=v.grad, log_theta=log_theta.grad)
    if not case["points"]:
        loss = ag.nll(g, case["kernel"], theta, v)
        loss.backward()
        return dict(nll=loss.detach(), v=v.grad, log_theta=log_theta.grad)
    pts = s["points"].detach().requires_grad_(True)
    loss = ag.nll(g, case["kernel"], theta, v, pts)
    loss.backward()
    return dict(nll=loss.detach(), v=v.grad, log_theta=log_theta.grad, points=pts.grad)


def work(case):
    N, k, path = case["N"], case["k"], case["path"]
    n0 = case["n0"] or min(N, max(k, 256))
    R = N - n0  # conditionals
    graph = R * (4 * k + 16)  # neighbour indices and coordinates
    pairs = k * (k + 1) // 2
    conditional = R * (22 * pairs + k ** 3 // 3 + 2 * k * k) + n0 ** 3 // 3
    apply = R * (2 * k + 2) + n0 * n0
    if path == "build":
        return dict(bytes=4 * N * case["d"] + 4 * N + 4 * R * k, flops=R * k * 8)
    if path == "factor":
        return dict(bytes=graph + R * (4 * k + 4) + 4 * n0 * n0, flops=conditional)
    if path == "sweep":
        return dict(bytes=2 * (R * (8 * k + 16) + 2 * n0 * n0), flops=2 * apply)
    if path == "vjp":
        return dict(bytes=2 * (R * (8 * k + 16) + 2 * n0 * n0) + 12 * N, flops=2 * apply)
    if path == "fly":
        return dict(bytes=2 * graph + 16 * N, flops=2 * (conditional + apply))
    back = R * (4 * k * k + 12 * pairs) + 2 * n0 ** 3
    if path == "fit":
        return dict(bytes=graph + 8 * N, flops=conditional + 2 * apply + back)
    stored = R * (4 * k + 4) + 2 * R * (8 * k + 16)
    return dict(bytes=graph + stored + 8 * N + (12 * N if case["points"] else 0),
                flops=conditional + 2 * apply + back * (2 if case["points"] else 1))


# ---- the same in plain torch, in 64 bits --------------------------------------
def _subtree(j, N):
    """Nodes of the left-balanced tree below (and with) node j, as a tensor."""
    lev = torch.zeros_like(j)
    for m in range(1, 40):
        lev += j + 1 >= 1 << m
    p = j - ((1 << lev) - 1)
    total = torch.zeros_like(j)
    for m in range(40):
        first = ((1 << m) - 1) + p
        fit = torch.div(N - first + (1 << lev) - 1, 1 << lev, rounding_mode="floor")
        fit = torch.minimum(fit, 1 << (m - lev).clamp(min=0))
        total += torch.where((m >= lev) & (first < N) & (j < N), fit, torch.zeros_like(fit))
    return total


def _tree(pts, N):
    """(tree index -> input index, tree index -> in-order rank): split on the
    widest extent, median by (coordinate, input index), children of node j of
    level l at j + 2^l and j + 2^(l+1)."""
    dev = pts.device
    tree_point = torch.zeros(N, dtype=torch.long, device=dev)
    inorder = torch.zeros(N, dtype=torch.long, device=dev)
    ids = torch.arange(N, device=dev)        # points not placed yet
    node = torch.zeros(N, dtype=torch.long, device=dev)   # the node they are below
    base = torch.zeros(N, dtype=torch.long, device=dev)   # in-order start of that node
    level = 0
    while len(ids):
        x = pts[ids]
        uniq, seg = torch.unique(node, return_inverse=True)
        S = len(uniq)
        ext = []
        for c in range(pts.shape[1]):
            lo = torch.full((S,), math.inf, device=dev).scatter_reduce(0, seg, x[:, c], "amin")
            hi = torch.full((S,), -math.inf, device=dev).scatter_reduce(0, seg, x[:, c], "amax")
            ext.append(hi - lo)
        dim = torch.zeros(S, dtype=torch.long, device=dev)
        best = ext[0]
        for c in range(1, len(ext)):
            dim = torch.where(ext[c] > best, torch.full_like(dim, c), dim)
            best = torch.maximum(best, ext[c])
        key = x.gather(1, dim[seg][:, None])[:, 0]
        # by (node, coordinate, input index); ids are in input order below each node
        o = torch.argsort(ids, stable=True)
        o = o[torch.argsort(key[o], stable=True)]
        o = o[torch.argsort(seg[o], stable=True)]
        ids, seg, node, base = ids[o], seg[o], node[o], base[o]
        start = torch.searchsorted(seg, torch.arange(S, device=dev))
        rank = torch.arange(len(ids), device=dev) - start[seg]
        left = _subtree(uniq + (1 << level), N)[seg]
        mid = rank == left
        tree_point[node[mid]] = ids[mid]
        inorder[node[mid]] = (base + left)[mid]
        right = rank > left
        node = torch.where(right, node + (2 << level), node + (1 << level))
        base = torch.where(right, base + left + 1, base)
        ids, node, base = ids[~mid], node[~mid], base[~mid]
        level += 1
    return tree_point, inorder


def _graph(case, pts):
    """The Vecchia graph: (order, coordinates by position in 64 bits,
    neighbour positions, level offsets, n0)."""
    N, k, dev = case["N"], case["k"], pts.device
    n0 = case["n0"] or min(N, max(k, 256))
    pts = torch.nn.functional.pad(pts + 0.0, (0, 3 - case["d"]))
    tree_point, inorder = _tree(pts, N)
    xt = pts[tree_point]
    nbr = torch.empty((N - n0, k), dtype=torch.long, device=dev)
    ix = torch.arange(N, device=dev)
    rows = max(1, min(2048, (1 << 28) // N))
    for a in range(n0, N, rows):
        e = min(N, a + rows)
        d2 = None
        for c in range(3):  # fma(dz, dz, fma(dy, dy, dx * dx)) in 32 bits
            df = (xt[:e, c][None, :] - xt[a:e, c][:, None]).double()
            df = df * df if d2 is None else df * df + d2
            d2 = df.float().double()
        key = (d2.float().view(torch.int32).long() << 32) | ix[:e][None, :]
        key = torch.where(ix[:e][None, :] < ix[a:e, None], key, torch.full_like(key, (1 << 63) - 1))
        nbr[a - n0:e - n0] = torch.topk(key, k, dim=1, largest=False, sorted=True).values & 0xffffffff
    depth = torch.zeros(N, dtype=torch.long, device=dev)
    while N > n0:
        new = depth[nbr].amax(1) + 1
        if torch.equal(new, depth[n0:]):
            break
        depth[n0:] = new
    o = torch.argsort(inorder, stable=True)
    o = o[torch.argsort(depth[o], stable=True)]  # position -> tree index
    pos = torch.empty_like(o)
    pos[o] = ix
    levels = [0] + torch.cumsum(torch.bincount(depth), 0).tolist()
    return tree_point[o], xt[o].double(), pos[nbr[o[n0:] - n0]], levels, n0


def _kappa(case, d2, ell, s2):
    if case["kernel"] == gg.SQEXP:
        return s2 * torch.exp(-0.5 * d2 / ell ** 2)
    zero = d2 == 0  # sqrt has no derivative there; kappa(0) = s2
    a = torch.sqrt(torch.where(zero, torch.ones_like(d2), d2)) / ell
    if case["kernel"] == gg.MATERN12:
        out = torch.exp(-a)
    elif case["kernel"] == gg.MATERN32:
        a = math.sqrt(3.0) * a
        out = (1.0 + a) * torch.exp(-a)
    else:
        a = math.sqrt(5.0) * a
        out = (1.0 + a + a * a / 3.0) * torch.exp(-a)
    return s2 * torch.where(zero, torch.ones_like(out), out)


def _conditional(case, x, nbr, at, ell, s2, nug):
    """b [R, k] and sigma^2 [R] of the positions `at` given their neighbours."""
    c = x[nbr]
    K = _kappa(case, (c[:, :, None, :] - c[:, None, :, :]).square().sum(-1), ell, s2)
    K = K + nug * torch.eye(nbr.shape[1], dtype=x.dtype, device=x.device)
    kc = _kappa(case, (c - x[at][:, None, :]).square().sum(-1), ell, s2)
    L = torch.linalg.cholesky(K)
    b = torch.cholesky_solve(kc[:, :, None], L)[:, :, 0]
    return b, s2 + nug - (b * kc).sum(1)


def _dense(case, x, n0, ell, s2, nug):
    K = _kappa(case, (x[:n0, None, :] - x[None, :n0, :]).square().sum(-1), ell, s2)
    return torch.linalg.cholesky(K + nug * torch.eye(n0, dtype=x.dtype, device=x.device))


def _chunks(n0, N, k):
    step = max(1, (1 << 25) // (k * k))
    return [(a, min(N, a + step)) for a in range(n0, N, step)]


def exact(case, seed):
    path, N, k = case["path"], case["N"], case["k"]
    if path == "build" or N > EXACT_MAX or N * k * k > (1 << 27) or case["rescue"]:
        return None  # whole numbers; out of reach; floored pivots
    s = _inputs(case, seed)
    order, x, nbr, levels, n0 = _graph(case, s["points"])
    if path in ("fit", "gradient"):
        return _exact_nll(case, s, order, x, nbr, n0)
    ell, s2, nug = case["ell"], 1.0, case["nugget"]
    parts = [_conditional(case, x, nbr[a - n0:e - n0], torch.arange(a, e, device=x.device), ell, s2,
                          nug) for a, e in _chunks(n0, N, k)]
    b = torch.cat([p[0] for p in parts]) if parts else x.new_zeros((0, k))
    L0 = _dense(case, x, n0, ell, s2, nug)
    sigma = torch.cat([L0.diagonal()] + [p[1].sqrt() for p in parts])
    logdet = 2.0 * sigma.log().sum().reshape(1)
    if path == "factor":
        return dict(b=b, sigma=sigma, L0=L0, logdet=logdet)
    xi = s["xi"].double()
    v = torch.empty_like(xi)
    v[:n0] = L0 @ xi[:n0]
    for a, e in zip(levels[1:-1], levels[2:]):
        v[a:e] = (b[a - n0:e - n0] * v[nbr[a - n0:e - n0]]).sum(1) + sigma[a:e] * xi[a:e]
    if path == "sweep":
        return dict(v=v, xi=xi, logdet=logdet)
    data = s["field"][order].double()
    if path == "fly":
        w0 = torch.linalg.solve_triangular(L0, data[:n0, None], upper=False)[:, 0]
        w = (data[n0:] - (b * data[nbr]).sum(1)) / sigma[n0:]
        return dict(v=v, nll=0.5 * (w0.square().sum() + w.square().sum() + logdet))
    u = v - data
    for a, e in reversed(list(zip(levels[1:-1], levels[2:]))):
        u.index_add_(0, nbr[a - n0:e - n0].reshape(-1),
                     (b[a - n0:e - n0] * u[a:e, None]).reshape(-1))
    return dict(v=v, xibar=torch.cat([L0.T @ u[:n0], sigma[n0:] * u[n0:]]))


def _exact_nll(case, s, order, x, nbr, n0):
    N, k, dev = case["N"], case["k"], x.device
    v = s["field"][order].double().requires_grad_(True)
    log_theta = s["log_theta"].double().to(dev).requires_grad_(True)
    x = x.requires_grad_(case["points"])
    total = 0.0
    for a, e in [(0, n0)] + _chunks(n0, N, k):
        ell, s2, nug = log_theta.exp()
        if a == 0:
            L0 = _dense(case, x, n0, ell, s2, nug)
            w = torch.linalg.solve_triangular(L0, v[:n0, None], upper=False)[:, 0]
            part = 0.5 * w.square().sum() + L0.diagonal().log().sum()
        else:
            n = nbr[a - n0:e - n0]
            b, var = _conditional(case, x, n, torch.arange(a, e, device=dev), ell, s2, nug)
            part = 0.5 * ((v[a:e] - (b * v[n]).sum(1)).square() / var + var.log()).sum()
        part.backward()
        total += float(part.detach())
    out = dict(nll=torch.tensor(total, dtype=torch.float64), v=v.grad, log_theta=log_theta.grad)
    if case["points"]:
        grad = torch.empty_like(x.grad)
        grad[order] = x.grad
        out["points"] = grad[:, :case["d"]].contiguous()
    return out
