"""Readouts into host memory.  Memory that nobody has written yet: the call faults every page in once, before the copy.  A page
that is read first faults twice (the shared zero page, then the write), and the copy into pages not faulted in is slower still.
Small states, which leave in one copy with their energies, and those just too large for it."""
import ctypes
import mmap
import resource

import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


def fresh(nbytes):
    m = mmap.mmap(-1, nbytes, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS)
    return m, np.frombuffer(m, np.float64)


def faults(call):
    f0 = resource.getrusage(resource.RUSAGE_SELF).ru_minflt
    assert call() == 0
    return resource.getrusage(resource.RUSAGE_SELF).ru_minflt - f0


def test_fresh_pages_fault_once():
    N, R, nT = 32, 4096, 16
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 31)]
    p = pkg.PT([N], Js, workload.geometric_ladder(0.3, 1.6, nT), R, 11, swap_every=0, measure_every=0, resync_every=0)
    a, E = p.state()  # the first call's own faults (driver, staging) are not counted
    H = p.energy()
    (ma, fa), (me, fe), (mh, fh) = fresh(a.nbytes), fresh(E.nbytes), fresh(E.nbytes)
    L, ptr = pkg.lib(), lambda x: ctypes.c_void_p(x.ctypes.data)
    pages = -(-(a.nbytes + E.nbytes) // mmap.PAGESIZE)
    assert pages >= 500
    # one fault a page; half of that again for whatever else the call faults in
    assert faults(lambda: L.pt_get_state(p._h, ptr(fa), ptr(fe))) <= 1.5 * pages
    assert L.pt_energy(p._h, ptr(fh)) == 0
    assert np.array_equal(fa, a.view(np.float64)) and np.array_equal(fe, E) and np.array_equal(fh, H)


@pytest.mark.parametrize("Ns,R,nT", [([256, 34], 12, 16), ([512], 1, 4), ([4, 96, 32], 2, 3), ([128], 2, 16), ([126, 128], 1, 16), ([4], 1, 1)],
                         ids=str)
def test_readout_of_few_chains(Ns, R, nT):
    """One copy up to 8192 words ([128] has 8224, [126, 128] 8160); the first ensemble in two pieces without measurements."""
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 40 + i) for i, N in enumerate(Ns)]
    temps = workload.geometric_ladder(0.3, 1.6, nT) if nT > 1 else [0.5]
    for prec in ("fp32", "fp64"):
        a, b = (pkg.PT(Ns, Js, temps, R, 5, precision=prec, swap_every=2, resync_every=0, measure_every=m) for m in (0, 1))
        for p in (a, b):
            p.sweep(4)
        (x, E), (y, F) = a.state(), b.state()
        assert np.array_equal(x, y) and np.array_equal(E, F)
        # the energies say which amplitudes belong to which place
        tol = 1e-5 if prec == "fp32" else 1e-12
        assert np.abs(a.energy() - E).max() <= tol * max(1.0, np.abs(E).max()) * max(Ns)
        a.set_state(np.conj(x))
        assert np.array_equal(a.state()[0], np.conj(x))
