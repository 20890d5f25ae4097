"""Readouts into host memory that nobody has written yet: the call faults every page in once, before the copy.  A page that is
read first faults twice (the shared zero page, then the write), and the copy into pages not faulted in is slower still."""
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
