// pt_rules.h -- index and scheduling arithmetic of the kernels and their launchers, free of CUDA so that a host compiler
// takes it too (tests/test_rules_host.py runs it at sizes no GPU test reaches).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define PT_HD __host__ __device__
#else
#define PT_HD
#endif

namespace ptgb {

// Warp of a thread counted over the grid.  64 bits: a block index times the block size passes 2^32 from 2^27 warps on, and
// a context may hold 2^28 chains.
PT_HD inline int64_t grid_warp(unsigned block, unsigned block_threads, unsigned thread) {
    return (int64_t)block * (block_threads / 32u) + thread / 32u;
}

// Tasks of one measurement of a (sample, temperature) with R replicas: the R chains, then the R (R - 1) / 2 replica pairs.
// From R = 65536 on they pass 2^31; with several measurements at once, earlier.
PT_HD inline int64_t measure_tasks(int R) { return R + (int64_t)R * (R - 1) / 2; }

// The at-th pair r1 < r2 of R replicas, in the order (0, 1), (0, 2), ..., (1, 2), ...  Row r starts at r (2R - r - 1) / 2; a few
// replicas are stepped through, for more the quadratic gives the row to within rounding.
PT_HD inline void replica_pair(int64_t at, int R, int *r1, int *r2) {
    auto row = [R](int64_t r) { return r * (2 * (int64_t)R - r - 1) / 2; };
    int64_t r = 0;
    if (R > 64) {
        const double b = 2.0 * R - 1.0, d = b * b - 8.0 * (double)at;
        r = (int64_t)(0.5 * (b - sqrt(d > 0.0 ? d : 0.0)));
        if (r > R - 2) r = R - 2;
        while (r > 0 && row(r) > at) --r;
    }
    while (row(r + 1) <= at) ++r;
    *r1 = (int)r;
    *r2 = (int)(r + 1 + (at - row(r)));
}

// Whether the full energies of comb chains run on the tiles of pt_energy.cu (FP32) or on blocks of (mode, block) items.  Tiles,
// but for small N with more groups than SMs: a tile block has an SM to itself and below N = 32 mostly waits, while 3 of the
// other fit (GB300, the kernel alone, 65536 chains: N = 4 66 us against 30, N = 16 131 against 68; 16384 chains of N = 32 73
// against 77; with few groups the tiles win at every N, N = 16, 160 chains 22 against 27 with its surroundings).
inline bool energy_tiles(bool fp64, int maxN, int groups, int sms) { return !fp64 && (maxN >= 32 || groups <= sms); }

// Thread blocks a group's full energy is split over, their partial sums added in a fixed order by a second kernel.  Items: about
// 8 blocks per SM (they wait on coupling loads).  Tiles: one block per SM at a time, so the number of parts that takes the
// least time in rounds of blocks: a block costs a + w / parts us, a for the group's tables, w for its tiles (fitted on GB300 to
// N = 4 ... 256 and groups of 8, 16 and 32: N = 16 a 2.2 ... 3, w 1 ... 4; N = 64 3.4 ... 5.9, 20 ... 56; N = 256, groups of 8, 25, 495).
constexpr int kEnergyPartsMax = 16;
inline int energy_parts(bool fp64, int maxN, int G, int groups, int sms) {
    if (!energy_tiles(fp64, maxN, groups, sms)) return std::max(1, std::min(8, (8 * sms + groups - 1) / std::max(groups, 1)));
    const double n2 = (double)maxN * maxN, a = 2.0 + n2 * (G + 8) / 48000.0, w = 4.0e-5 * n2 * std::sqrt((double)maxN) * (G + 4);
    double best = 1e300;
    int parts = 1;
    for (int q = 1; q <= kEnergyPartsMax; ++q) {
        const double t = (double)(((int64_t)groups * q + sms - 1) / sms) * (a + w / q);
        if (t < best) { best = t; parts = q; }
    }
    return parts;
}

// Work units (group, run) of a persistent sweep launch are counted in 32 bits: the runs are as few as that takes.
constexpr int64_t kUnitsMax = 1 << 30;

// Sweeps of a unit where units are whole sweeps: those asked for, more where seg sweeps of that many groups make too many units.
inline int unit_sweeps(int seg, int sweeps, int groups) {
    const int64_t runs = std::max<int64_t>(1, kUnitsMax / std::max(groups, 1));
    return (int)std::min<int64_t>(seg, std::max<int64_t>(sweeps, (seg + runs - 1) / runs));
}

// Runs each group's updates are cut into on a device that holds `most` groups at once: those that leave the least of the last
// round of units idle.  A unit costs about 8 us beside its updates (tables, amplitudes, the first couplings), an update of
// the largest N about 2 + N^2 / 6000 us (GB300).  Measured there against one run per group and sweep (192 groups of
// N = 256 on 152 SMs): 2298 -> 2127 us per sweep at 8 sweeps a launch, where the second round left 112 SMs idle.
// A run is no longer than about kUnitUs, however many sweeps the launch has: in a ragged ensemble the next run of a large group
// may be taken up while the one before still works, and that wait gives up after 10 s (kWaitNs).  Groups that all fit at once
// keep one run, which nobody waits for.
constexpr double kUnitUs = 1e6;
inline int sweep_runs(int groups, int most, int64_t updates, int maxN) {
    if (groups <= most) return 1;
    const double group_us = (double)updates * (2.0 + maxN * (double)maxN / 6000.0);
    const int64_t cap = std::max<int64_t>(1, std::min<int64_t>(updates, kUnitsMax / std::max(groups, 1)));
    const int64_t least = std::min<int64_t>(cap, 1 + (int64_t)(group_us / kUnitUs)), top = std::min<int64_t>(cap, std::max<int64_t>(512, 2 * least));
    int64_t best = least;
    double best_t = 1e300;
    for (int64_t k = least; k <= top; ++k) {
        const int64_t rounds = std::max<int64_t>(k, ((int64_t)groups * k + most - 1) / std::max(most, 1));  // runs of a group queue up
        const double t = (double)rounds * (group_us / (double)k + 8.0);
        if (t < best_t) { best_t = t; best = k; }
    }
    return (int)best;
}

// Whether amplitudes and energies (words of 8 bytes in all) come to the host in one copy and are handed out from it: while they are
// few, a copy saved is worth more than the pass over host memory.  GB300, us a call of 4 chains, one copy / two / with the order put
// right on the host instead of by a launch: N = 18 36 / 48 / 43, N = 64 37 / 50 / 44, N = 512 42 / 52 / 46.
inline bool state_in_one_copy(size_t words) { return words <= 8192; }

// Bytes of the snapshot buffer: n_snap states of the chains (pairs of reals).  A host readout passes through it widened to FP64, in
// as many pieces as that takes; FP32 with one snapshot would need two, which costs a small state more than the copy itself
// (N = 64, 12 chains: 72 us against 46 in one piece; N = 256, 96 chains: 98 against 65, on GB300), so up to 1 MB it has the room.
inline size_t snapshot_bytes(int n_snap, int64_t a_total, size_t real_bytes) {
    const size_t wide = (size_t)a_total * 16;
    return std::max((size_t)n_snap * (size_t)a_total * 2 * real_bytes, std::min(wide, (size_t)1 << 20));
}

}  // namespace ptgb
