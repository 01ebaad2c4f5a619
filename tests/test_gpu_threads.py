"""Several host threads, each with its own graph, factor and stream, at sizes that
ask one kernel for different amounts of shared memory (dense blocks, the runs of
small levels): the calls succeed and give what one thread alone gets."""
import threading

import pytest
import torch

import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import to_gpu

pytestmark = pytest.mark.gpu

SIZES = [(500, 4, 64), (9000, 16, 300), (40000, 16, 320), (20000, 16, 200)]
KERN = gg.Kernel(gg.MATERN32, 1.0, 0.2, 1e-3)


def work(pts, xi, k, n0, reps):
    out = []
    g = gg.build_graph(pts, k, n0=n0)
    for _ in range(reps):
        f = gg.factor(g, KERN)
        v = gg.generate(g, f, xi)
        xb, _ = gg.generate_backward(g, f, xi, v, xi, theta=False)
        out.append((v, gg.whiten(g, f, v), xb))
    torch.cuda.current_stream().synchronize()
    assert gg.sync_status(g)[0] == 0
    return out


def test_threads_with_different_sizes():
    data = [(to_gpu(workloads.uniform_cube(N, N)), to_gpu(workloads.white_noise(N, 1)), k, n0)
            for N, k, n0 in SIZES]
    torch.cuda.synchronize()
    alone = [work(*d, 1)[0] for d in data]
    got, errors = [None] * len(data), []

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                got[i] = work(*data[i], 20)
        except Exception as e:  # noqa: BLE001
            errors.append((i, e))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(data))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for ref, mine in zip(alone, got):
        for v, xi, xb in mine:
            assert torch.equal(v, ref[0]) and torch.equal(xi, ref[1])
            assert (xb - ref[2]).norm() <= 1e-6 * ref[2].norm()  # atomic sums, any order
