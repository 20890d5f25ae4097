"""Index and scheduling arithmetic of the kernels (csrc/pt_rules.h), compiled by the host compiler and run at sizes that no
GPU test reaches."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "pt_rules.h"
using namespace ptgb;
extern "C" {
int64_t grid_warp_(unsigned b, unsigned n, unsigned t) { return grid_warp(b, n, t); }
int64_t measure_tasks_(int R) { return measure_tasks(R); }
void replica_pair_(int64_t at, int R, int *r1, int *r2) { replica_pair(at, R, r1, r2); }
int unit_sweeps_(int seg, int sweeps, int groups) { return unit_sweeps(seg, sweeps, groups); }
int sweep_runs_(int groups, int most, int64_t updates, int maxN) { return sweep_runs(groups, most, updates, maxN); }
int64_t snapshot_bytes_(int n, int64_t a, int real) { return (int64_t)snapshot_bytes(n, a, (size_t)real); }
int energy_parts_(int fp64, int maxN, int G, int groups, int sms) { return energy_parts(fp64, maxN, G, groups, sms); }
int energy_tiles_(int fp64, int maxN, int groups, int sms) { return energy_tiles(fp64, maxN, groups, sms); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "librules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2511_13508_gb300", "csrc"),
                    str(d / "shim.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.grid_warp_.restype = L.measure_tasks_.restype = ctypes.c_int64
    L.snapshot_bytes_.argtypes, L.snapshot_bytes_.restype = [ctypes.c_int, ctypes.c_int64, ctypes.c_int], ctypes.c_int64
    L.sweep_runs_.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    L.replica_pair_.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.POINTER(ctypes.c_int), ctypes.POINTER(ctypes.c_int)]
    return L


@pytest.mark.parametrize("chain", [0, 7, 8, (1 << 27) - 1, 1 << 27, (1 << 27) + 9, (1 << 28) - 1])
def test_a_warp_per_chain_reaches_every_chain(rules, chain):
    """Blocks of 8 warps: chain c is warp c of the grid, up to the 2^28 chains of a context."""
    for lane in (0, 31):
        assert rules.grid_warp_(chain // 8, 256, chain % 8 * 32 + lane) == chain


def _pair(rules, at, R):
    a, b = ctypes.c_int(), ctypes.c_int()
    rules.replica_pair_(at, R, ctypes.byref(a), ctypes.byref(b))
    return a.value, b.value


@pytest.mark.parametrize("R", [2, 3, 63, 64, 65, 66, 130])
def test_replica_pairs_come_in_order(rules, R):
    pairs = [(i, j) for i in range(R) for j in range(i + 1, R)]
    assert rules.measure_tasks_(R) == R + len(pairs)
    assert [_pair(rules, n, R) for n in range(len(pairs))] == pairs


@pytest.mark.parametrize("R", [46340, 46341, 65535, 65536, 70000, (1 << 24) + 1, 1 << 28])
def test_replica_pairs_of_very_many_replicas(rules, R):
    """Where the count of pairs passes 2^31, up to the largest ensemble: ends, row ends and rows in the middle."""
    n = R * (R - 1) // 2
    assert rules.measure_tasks_(R) == R + n
    assert _pair(rules, 0, R) == (0, 1) and _pair(rules, n - 1, R) == (R - 2, R - 1)
    for r in (1, 2, R // 3, R // 2, R - 40, R - 3):
        at = r * (2 * R - r - 1) // 2
        assert _pair(rules, at, R) == (r, r + 1) and _pair(rules, at - 1, R) == (r - 1, R - 1)


@pytest.mark.parametrize("seg,sweeps,groups", [(64, 1, 192), (64, 8, 1), (7, 32, 5000), (1 << 20, 1, 5000), (1 << 28, 1, 12),
                                               (1 << 29, 3, 1), (64, 1, 1 << 25), (1 << 20, 1, 1 << 25)])
def test_units_of_a_launch_fit_32_bits(rules, seg, sweeps, groups):
    unit = rules.unit_sweeps_(seg, sweeps, groups)
    assert 1 <= unit <= seg and unit >= min(seg, sweeps)
    units = -(-seg // unit) * groups
    assert units <= 1 << 30
    if -(-seg // sweeps) * groups <= 1 << 30:
        assert unit == min(seg, sweeps)


@pytest.mark.parametrize("groups", [1, 152, 160, 192, 5000, 1 << 20, 3 << 20, 1 << 23, 1 << 25])
@pytest.mark.parametrize("updates,N", [(2, 4), (224, 64), (8192, 256), (1 << 30, 64)])
def test_runs_of_a_launch_fit_32_bits(rules, groups, updates, N):
    runs = rules.sweep_runs_(groups, 152, updates, N)
    assert 1 <= runs <= updates and runs * groups <= 1 << 30
    if groups <= 152:
        assert runs == 1


@pytest.mark.parametrize("n,a,real,pieces", [(1, 2, 4, 1), (1, 768, 4, 1), (1, 65536, 4, 1), (1, 65538, 4, 2), (1, 1 << 30, 4, 2),
                                             (2, 1 << 30, 4, 1), (5, 18, 4, 1), (1, 16, 8, 1), (1, 1 << 30, 8, 1)])
def test_snapshots_hold_a_readout(rules, n, a, real, pieces):
    """A state of a FP64 pairs passes through the snapshot buffer in this many pieces."""
    room = rules.snapshot_bytes_(n, a, real)
    assert room >= n * a * 2 * real and -(-a // (room // 16)) == pieces


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("N", [4, 16, 30, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("G", [8, 16, 32])
def test_parts_of_a_full_energy(rules, fp64, N, G):
    """Any number of groups has a valid number of parts; FP32 tiles of small N are not split where the groups fill the SMs
    anyway (a block's tables cost more than its share of the tiles), few groups are split to fill them."""
    for groups in (1, 3, 100, 152, 153, 160, 256, 2048, 1 << 25):
        q = rules.energy_parts_(fp64, N, G, groups, 152)
        assert 1 <= q <= (16 if rules.energy_tiles_(fp64, N, groups, 152) else 8)
        if not fp64 and groups == 256 and 32 <= N <= 64:
            assert q <= 2
        if groups == 1:
            assert q == (16 if not fp64 else 8)
    assert rules.energy_tiles_(fp64, N, 152, 152) == (not fp64) and rules.energy_tiles_(fp64, N, 153, 152) == (not fp64 and N >= 32)


@pytest.mark.parametrize("N,sweeps", [(48, 3), (64, 7), (64, 3), (128, 7)])
def test_a_few_groups_too_many_are_cut_inside_sweeps(rules, N, sweeps):
    """160 groups on 152 SMs, launches of test_gpu_comb_runs: runs whose ends are no ends of sweeps."""
    runs = rules.sweep_runs_(160, 152, sweeps * N // 2, N)
    assert runs > 1 and sweeps % runs


@pytest.mark.parametrize("groups,most", [(153, 152), (192, 152), (5000, 152), (40, 8)])
@pytest.mark.parametrize("updates,N", [(1 << 30, 64), (1 << 30, 256), (100000 * 128, 256), (1 << 30, 512), (20, 4)])
def test_a_run_is_short_beside_the_bound_on_waits(rules, groups, most, updates, N):
    """A unit waits 10 s at most for the run before it, so a run stays near a second (an update 2 + N^2 / 6000 us)."""
    runs = rules.sweep_runs_(groups, most, updates, N)
    assert 1 <= runs <= updates and runs * groups <= 1 << 30
    assert updates / runs * (2 + N * N / 6000) <= 1.01e6
