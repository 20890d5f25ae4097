"""Executed flop count of a sweep where a chain keeps its pair products (one chain per block): coupling terms and field rows
alone, against a count over the quadruplet list."""
import pytest

import bench


@pytest.mark.parametrize("N", [4, 6, 10, 16])
def test_flops_without_pair_products_match_the_quadruplets(N):
    quads = [(a, b, c, b + c - a) for a in range(N) for b in range(a + 1, N) for c in range(b + 1, N) if b + c - a < N]
    terms = [0] * N  # couplings of every mode's field
    rows = [set() for _ in range(N)]  # partners m with a pair of the sum l + m
    for a, b, c, d in quads:
        for l, m in ((a, d), (d, a), (b, c), (c, b)):
            terms[l] += 1
            rows[l].add(m)
    # N / 2 updates of an ordered pair of distinct modes, each mode in 2 / N of them
    want = sum(4.0 * terms[l] + 8.0 * len(rows[l]) for l in range(N))
    assert bench.flops_per_chain_sweep(N, products=False) == pytest.approx(want, rel=1e-12)
    assert bench.flops_per_chain_sweep(N) > bench.flops_per_chain_sweep(N, products=False)
