"""Creation with less device memory than the fastest kernels want.  What a context cannot do without is allocated first; the
stores of the faster sweeps (pair-table lists of a graph, row store of the comb) come last, are left out when they do not fit
and are then given back whole, so that whatever fits without them is created and runs on the other kernels.

The allocator callbacks count bytes and refuse what passes a limit; no allocation of the device fails.
"""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


class Budget(pkg._TorchAllocator):
    """The binding's allocator with a limit on the bytes it has out."""

    def __init__(self, stream, limit):
        super().__init__(stream)
        self.limit, self.sizes = limit, {}
        alloc, free = self.alloc, self.free

        def _alloc(nbytes, user):
            if self.live + nbytes > self.limit:
                return None
            p = alloc(nbytes, user)
            if p:
                self.sizes[p] = nbytes
            return p

        def _free(ptr, user):
            self.sizes.pop(ptr)
            free(ptr, user)

        self._keep = (alloc, free)
        self.alloc, self.free = pkg.ALLOC_FN(_alloc), pkg.FREE_FN(_free)

    @property
    def live(self):
        return sum(self.sizes.values())


@pytest.fixture
def create(monkeypatch):
    """create(limit, ...) -> (context or None when it does not fit, bytes it holds)"""
    made = []

    def one(limit, *args, **kw):
        def allocator(stream):
            made.append(Budget(stream, limit))
            return made[-1]
        monkeypatch.setattr(pkg, "_TorchAllocator", allocator)
        try:
            p = pkg.PT(*args, **kw)
        except pkg.PTError as e:
            assert e.code == -2 and made[-1].live == 0, (e, made[-1].live)
            return None, 0
        return p, made[-1].live
    return one


def same_run(a, b, n, tol):
    for p in (a, b):
        p.sweep(n)
    (x, E), (y, F) = a.state(), b.state()
    assert np.abs(x - y).max() <= tol and np.abs(E - F).max() <= tol * max(1.0, np.abs(F).max())


ALL = 1 << 62


def test_graph_lists_give_way(create):
    N = 32
    g = [pkg.fmc_graph(workload.random_frequencies(N, 300 + i)) for i in range(3)]
    Js = [workload.couplings(N, len(x), 60 + i) for i, x in enumerate(g)]
    args = ([N] * 3, Js, workload.geometric_ladder(0.3, 1.6, 5), 2, 29)
    kw = dict(precision="fp32", graphs=g, swap_every=0, measure_every=2, resync_every=0)
    full, need = create(ALL, *args, **kw)
    lists = sum(6 * 16 * len(x) for x in g)  # the quadruplets of every pair of modes alone
    for lack in (256, lists // 2, lists):  # the last list does not fit, the cross lists, the first list
        p, held = create(need - lack, *args, **kw)
        assert p is not None and held <= need - lists, (lack, held, need)
        same_run(p, create(ALL, *args, **dict(kw, precision="fp64_plain"))[0], 3, 1e-5)
        least = held
    p, held = create(least, *args, **kw)
    assert p is not None and held == least
    assert create(least - 256, *args, **kw)[0] is None


@pytest.mark.parametrize("prec,N,G", [("fp64", 66, 16), ("fp64", 24, 16), ("fp64", 160, 8), ("fp32", 24, 16)])
def test_row_store_gives_way(create, prec, N, G):
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 5)]
    args = ([N], Js, workload.geometric_ladder(0.3, 1.6, 5), 2, 17)
    kw = dict(precision=prec, swap_every=2, measure_every=2, resync_every=0)
    block, base = create(ALL, *args, **dict(kw, chains_per_block=G))
    full, need = create(ALL, *args, **kw)
    # beside what the J-sharing blocks hold, a context keeps the row store and the order of its chains
    row = N * (N // 2) * N * (8 if prec == "fp64" else 4)
    assert base + row <= need <= base + row + 1024, (need - base, row)
    for lack in (256, row // 2, row):
        p, held = create(need - lack, *args, **kw)
        assert p is not None and held == base, (lack, held, base)
        same_run(p, block if lack == 256 else create(ALL, *args, **dict(kw, chains_per_block=G))[0], 3, 1e-12 if prec == "fp64" else 1e-5)
    p, held = create(base, *args, **kw)
    assert p is not None and held == base
    assert create(base - 256, *args, **kw)[0] is None
    same_run(full, create(ALL, *args, **kw)[0], 3, 0.0)


def test_partial_energies_follow_the_groups(create):
    """Partial sums of the full energy take 256 bytes per group and part; an FP64 ensemble of 1024 groups of 8 has two parts, and
    the state, its snapshot and the books of a chain of 4 modes stay below 330 bytes."""
    Js = [workload.couplings(4, 1, 5)]
    p, held = create(ALL, [4], Js, [0.5, 1.0], 4096, 17, precision="fp64", chains_per_block=8, swap_every=0, measure_every=0)
    assert held <= 8192 * (330 + 64), held / 8192
    p.resync()
    assert np.isfinite(p.energy()).all()
