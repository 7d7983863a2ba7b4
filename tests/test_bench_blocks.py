"""The benchmark's flop count of the symmetric CUDA-core stage against an
independent count of the node orbits.  No GPU."""
import itertools

import pytest

import bench

V4 = [(0, 1, 2, 3), (1, 0, 3, 2), (2, 3, 0, 1), (3, 2, 1, 0)]


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_block_flops_follow_the_orbits(N):
    nodes = [b for b in itertools.product(range(N + 1), repeat=4) if sum(b) == N]
    orbits = {frozenset(tuple(b[i] for i in g) for g in V4) for b in nodes}
    free = sum(len(o) == 4 for o in orbits)
    # an orbit carries the first character once; a free one every other character,
    # one of two nodes one of the three others
    D0 = len(orbits)
    D1 = free + sum(len(o) == 2 for o in orbits) // 3
    Np, Nfp = len(nodes), (N + 1) * (N + 2) // 2
    assert D0 + 3 * D1 == Np
    # blocks of d/dxi_a: D0 x D1, D1 x D0 and two D1 x D1 for each direction
    D = 3 * (2 * D0 * D1 + 2 * D1 * D1)
    for fp64 in (False, True):
        f, g = bench.block_flops(N, Np, Nfp, 10, 4, False, fp64)
        rest = (36 if fp64 else 72) * Np + 12 * Nfp * Np + 48 * Np + 288 * Nfp
        assert f == (8 if fp64 else 12) * D + rest
        # a rule of half the symmetry: twice the coefficients per group
        g2 = bench.block_flops(N, Np, Nfp, 10, 2, False, fp64)[1]
        assert g2 - g == 48 * Np * 10
        assert f < bench.algorithmic_costs(N, Np, Nfp, 40, 4, False)["flops_std"] or N == 1
