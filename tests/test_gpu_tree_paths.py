"""The tree where its way through the levels changes: subtrees that just fit one
block (1024 nodes) or just do not, with full and ragged last levels; the sizes
where the partitions of a level stop sharing a launch.  Bit for bit against the
oracle, both split rules, with ties, duplicates and flat clouds."""
import numpy as np
import pytest

import oracle
import paper_2606_11402_gb300 as gg
import workloads
from gpu_util import np_, to_gpu

pytestmark = pytest.mark.gpu


def points(kind, N):
    x = workloads.uniform_cube(N, N)
    if kind == "ties":  # coordinates on a coarse grid, many points equal
        x = np.round(x * 6) / 6
    if kind == "flat":
        x[:, 1] = 0.25
    return x


def check(x, rule):
    g = gg.build_graph(to_gpu(x), 1, n0=1, split_rule=rule)
    tp, sd, io, _, _ = g.export_tree()
    for got, want in zip((tp, sd, io), oracle.tree_build(oracle.canonicalise(x), rule)):
        assert np.array_equal(np_(got), want)


@pytest.mark.parametrize("N", [2, 3, 31, 33, 1022, 1023, 1024, 1025, 2046, 2047, 2048, 2049, 2050,
                               3071, 3072, 4097, 65535, 65536, 131073])
@pytest.mark.parametrize("kind", ["uniform", "ties", "flat"])
@pytest.mark.parametrize("rule", [0, 1])
def test_tree_edges(N, kind, rule):
    check(points(kind, N), rule)


@pytest.mark.parametrize("N", [1 << 21, (1 << 21) + 1])
def test_tree_batch_line(N):
    check(points("uniform", N), 0)
