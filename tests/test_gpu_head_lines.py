"""generate where the run of levels that one block takes ends: by row entries a level,
with more of them when the block finishes the cloud; row slices of 28 entries, which
have half the threads; few large levels (k = 1), which go behind the barrier."""
import pytest

import workloads
from test_gpu_sweep_paths import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 8, 12, 16, 20, 24, 25, 28, 32, 48, 64])
@pytest.mark.parametrize("N", [900, 4096, 10007, 30011])
def test_small_clouds(N, k):
    check(workloads.unit_gaussian(N, N + k), k, 100)


@pytest.mark.parametrize("N,k", [(2_000_000, 1), (400_000, 28), (500_000, 12)])
def test_larger_clouds(N, k):
    check(workloads.unit_gaussian(N, k), k, 256)
