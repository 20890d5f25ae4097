// pt_aux.cu -- chain initialisation, replica-exchange swaps, measurements and the plain FP64 path of
// the smoothed-cubic Parallel-Tempering engine (arXiv 2511.13508).
#include <cstdint>
#include "pt_common.cuh"
#include "pt_kernels.h"
#include "pt_rules.h"

namespace ptgb {

template <typename T> __device__ __forceinline__ T block_sum(T v, T *scratch) {
    // scratch: >= 32 entries; every thread of the block must call
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = (blockDim.x + 31) / 32;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    T t = T(0);
    for (int w = 0; w < nw; ++w) t += scratch[w];
    return t;
}

// ------------------------------------------------------------------------------------------------
// Initial chains: exact draws of the beta = 0 law (uniform on sum |a|^4 = N with uniform phases):
// u = sqrt(N) |g| / ||g||, g Gaussian by Box-Muller, a_k = sqrt(u_k) e^{i phi_k}.  Stream INIT with
// counter (chain id, mode, 0, tag), chain id = (s R + r) nT + t.
__global__ void init_kernel(InitParams p) {
    __shared__ double scratch[32];
    const int slot = blockIdx.x;
    const int s = p.chain_sample[slot];
    const SampleDev sd = p.samples[s];
    const int N = sd.N;
    const int r = (slot - sd.chain0) / p.nT, t = p.label[slot];
    const uint32_t cid = (uint32_t)((s * p.R + r) * p.nT + t);
    double g2 = 0.0;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        const u32x4 w = draw(p.seed, cid, (uint32_t)k, 0u, kTagInit);
        const double g = sqrt(-2.0 * log(u01(w.x))) * cos(kTwoPi * u01(w.y));
        g2 += g * g;
    }
    const double nrm = sqrt(block_sum(g2, scratch));
    const int64_t base = sd.a_off + (int64_t)(slot - sd.chain0) * N;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        const u32x4 w = draw(p.seed, cid, (uint32_t)k, 0u, kTagInit);
        const double g = sqrt(-2.0 * log(u01(w.x))) * cos(kTwoPi * u01(w.y));
        const double ph = kTwoPi * u01(w.z);
        const double u = sqrt((double)N) * fabs(g) / nrm;
        const double A = sqrt(u);
        const double re = A * cos(ph), im = A * sin(ph);
        if (p.dbl) reinterpret_cast<double2 *>(p.a)[base + k] = make_double2(re, im);
        else reinterpret_cast<float2 *>(p.a)[base + k] = make_float2((float)re, (float)im);
    }
}

cudaError_t launch_init(const InitParams &p, int n_chains, cudaStream_t s) {
    if (n_chains <= 0) return cudaSuccess;
    init_kernel<<<n_chains, 128, 0, s>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// Canonical order: chain slot -> (sample, replica, temperature its label names).  One warp per chain.
template <typename V>
__global__ void canon_kernel(const SampleDev *samples, const int *chain_sample, const int *label, int nT, const V *a, double2 *a_out,
                             int64_t lo, int64_t hi, const double *E, double *E_out, int n_chains) {
    const int64_t warp = grid_warp(blockIdx.x, blockDim.x, threadIdx.x);
    if (warp >= n_chains) return;
    const int slot = (int)warp, lane = threadIdx.x & 31;
    const SampleDev sd = samples[chain_sample[slot]];
    const int at = (slot - sd.chain0) / nT * nT + label[slot];
    if (E && lane == 0) E_out[sd.chain0 + at] = E[slot];
    if (!a) return;
    const V *src = a + sd.a_off + (int64_t)(slot - sd.chain0) * sd.N;
    const int64_t dst = sd.a_off + (int64_t)at * sd.N;
    for (int x = lane; x < sd.N; x += 32) {
        if (dst + x < lo || dst + x >= hi) continue;
        const V v = src[x];
        a_out[dst + x - lo] = make_double2((double)v.x, (double)v.y);
    }
}

cudaError_t launch_canon(const SampleDev *samples, const int *chain_sample, const int *label, int nT, const void *a, bool dbl,
                         double2 *a_out, int64_t lo, int64_t hi, const double *E, double *E_out, int n_chains, cudaStream_t s) {
    const int grid = (n_chains + 7) / 8;
    if (dbl) canon_kernel<double2><<<grid, 256, 0, s>>>(samples, chain_sample, label, nT, (const double2 *)a, a_out, lo, hi, E, E_out, n_chains);
    else canon_kernel<float2><<<grid, 256, 0, s>>>(samples, chain_sample, label, nT, (const float2 *)a, a_out, lo, hi, E, E_out, n_chains);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// One swap pass: per (sample, replica) ladder, sequentially i = 0 .. nT-2 (ascending T), exchange the
// temperatures of the chains at i and i+1 with probability min[1, exp((b_i - b_{i+1})(E_i - E_{i+1}))]
// (paper Eq. (15)).  Labels are exchanged instead of configurations.  The per-chain Metropolis
// counters are first folded into per-temperature counters under the labels they were earned with.
// One warp per ladder.  The sequence is a chain of FP64 operations, so everything else is taken off it: chains, energies
// and counters are loaded by all lanes, and the uniforms are drawn as log U, a lane each, so that a step is a difference,
// a product and a comparison (it used to hold an exponential and three dependent loads: 78 us for a ladder of 42
// temperatures on GB300).
constexpr int kSwapTile = 256;  // temperatures of a ladder handled at once

__global__ void __launch_bounds__(32) swap_kernel(SwapParams p) {
    __shared__ double sE[kSwapTile + 1], sB[kSwapTile + 1], sL[kSwapTile];
    __shared__ int sC[kSwapTile + 1], sS[kSwapTile];
    const int ladder = blockIdx.x, lane = threadIdx.x, s = ladder / p.R;
    int *perm = p.perm + (int64_t)ladder * p.nT;
    const uint32_t pass = (uint32_t)p.ctl->swap_passes;
    const int64_t pair0 = (int64_t)ladder * (p.nT - 1);
    for (int i0 = 0; i0 == 0 || i0 + 1 < p.nT; i0 += kSwapTile) {
        const int n = min(kSwapTile, p.nT - 1 - i0);  // pairs (i, i+1) of this tile
        for (int i = lane; i <= n; i += 32) {
            const int slot = perm[i0 + i];
            sC[i] = slot;
            sE[i] = p.E[slot];
            sB[i] = p.beta[i0 + i];
            if (i < n) sL[i] = log(u01(draw(p.seed, (uint32_t)ladder, pass, (uint32_t)(i0 + i), kTagSwap).x));
            if (i > 0 || i0 == 0) {  // entry 0 of a later tile is the last of the one before: folded there
                atomicAdd(p.mcT_acc + (int64_t)s * p.nT + i0 + i, p.mc_acc[slot]);
                atomicAdd(p.mcT_att + (int64_t)s * p.nT + i0 + i, p.mc_att[slot]);
                p.mc_acc[slot] = 0ull;
                p.mc_att[slot] = 0ull;
            }
        }
        __syncwarp();
        if (n > 0) {
            int c0 = sC[0];
            double e0 = sE[0];
            for (int i = 0; i < n; ++i) {
                const double e1 = sE[i + 1], D = (sB[i] - sB[i + 1]) * (e0 - e1);
                const bool swap = D >= 0.0 || sL[i] < D;
                const int c1 = sC[i + 1];
                // position i keeps the chain that does not move on
                if (lane == 0) { sC[i] = swap ? c1 : c0; sS[i] = swap; }
                if (!swap) { c0 = c1; e0 = e1; }
            }
            if (lane == 0) sC[n] = c0;
        }
        __syncwarp();
        for (int i = lane; i <= n; i += 32) {
            perm[i0 + i] = sC[i];
            p.label[sC[i]] = i0 + i;
            if (i < n) {
                p.swap_att[pair0 + i0 + i] += 1ull;
                if (sS[i]) p.swap_acc[pair0 + i0 + i] += 1ull;
            }
        }
        __syncwarp();
        __threadfence_block();
    }
}

// Many ladders of at most L temperatures, L lanes each: the same steps on values that the lanes hold, exchanged by shuffles.  A
// warp per ladder leaves nearly all lanes idle there (GB300, us per pass with a thread per ladder that takes every step alone / a
// warp / here: 4000 ladders of 2 temperatures 15 / 19 / 14, 100000 171 / 231 / 136, 10000 of 3 29 / 35 / 24; 100 of 3 11 / 10 /
// 13, so few ladders keep their warps; from 5 temperatures on the warp beats the thread at every count, 10000 ladders 40 / 45).
constexpr int kSwapShort = 4, kSwapMany = 2000;

template <int L> __global__ void __launch_bounds__(128) swap_short_kernel(SwapParams p) {
    const int64_t ladder = ((int64_t)blockIdx.x * 128 + threadIdx.x) / L;
    const int i = threadIdx.x % L, s = (int)(ladder / p.R);
    const bool mine = ladder < (int64_t)p.S * p.R && i < p.nT;  // the others only take part in the shuffles
    int *perm = p.perm + ladder * p.nT;
    const int64_t pair = ladder * (p.nT - 1) + i;
    int slot = 0;
    double E = 0.0, b = 0.0, lu = 0.0;
    if (mine) {
        slot = perm[i];
        E = p.E[slot];
        b = p.beta[i];
        if (i + 1 < p.nT) lu = log(u01(draw(p.seed, (uint32_t)ladder, (uint32_t)p.ctl->swap_passes, (uint32_t)i, kTagSwap).x));
        atomicAdd(p.mcT_acc + (int64_t)s * p.nT + i, p.mc_acc[slot]);
        atomicAdd(p.mcT_att + (int64_t)s * p.nT + i, p.mc_att[slot]);
        p.mc_acc[slot] = 0ull;
        p.mc_att[slot] = 0ull;
    }
    const unsigned all = 0xffffffffu;
    int c0 = __shfl_sync(all, slot, 0, L), kept = slot;
    double e0 = __shfl_sync(all, E, 0, L);
    bool swapped = false;
    for (int k = 0; k + 1 < p.nT; ++k) {
        const int c1 = __shfl_sync(all, slot, k + 1, L);
        const double e1 = __shfl_sync(all, E, k + 1, L), db = __shfl_sync(all, b, k, L) - __shfl_sync(all, b, k + 1, L);
        const double D = db * (e0 - e1);
        const bool swap = D >= 0.0 || __shfl_sync(all, lu, k, L) < D;
        if (i == k) { kept = swap ? c1 : c0; swapped = swap; }
        if (!swap) { c0 = c1; e0 = e1; }
    }
    if (!mine) return;
    if (i + 1 == p.nT) kept = c0;
    perm[i] = kept;
    p.label[kept] = i;
    if (i + 1 < p.nT) {
        p.swap_att[pair] += 1ull;
        if (swapped) p.swap_acc[pair] += 1ull;
    }
}

template <int L> static cudaError_t launch_swap_short(const SwapParams &p, int n, cudaStream_t s) {
    swap_short_kernel<L><<<(unsigned)(((int64_t)n * L + 127) / 128), 128, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_swap(const SwapParams &p, cudaStream_t s) {
    const int n = p.S * p.R;
    if (n <= 0 || p.nT < 2) return cudaSuccess;
    if (n > kSwapMany && p.nT <= 2) return launch_swap_short<2>(p, n, s);
    if (n > kSwapMany && p.nT <= kSwapShort) return launch_swap_short<kSwapShort>(p, n, s);
    swap_kernel<<<n, 32, 0, s>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// Measurements of one (sample, temperature) per block over the snapshots and/or the live state:
// E, E^2 (specific heat, Eq. (21)), Y2, Y4 (Sec. IV.D), I, I^2 per chain; for every replica pair the
// overlap q = Re sum conj(a^c) a^d / N (Sec. IV.C), its moments and its 201-bin histogram.
// A task (one chain, or one pair of replicas, of one measurement) is one warp's; the sums over tasks are then taken in
// task order, one thread per accumulator.  (One block per chain and pair in turn, with block-wide reductions: 103 us for
// 5 measurements of 4 replicas at N = 18 on GB300, latency of the reductions.)
constexpr int kMeasWarps = 8, kMeasBatch = 32;

// I counts the tasks: int, or int64_t where all measurements together have more than 2^30.
template <typename V, typename I> __global__ void __launch_bounds__(kMeasWarps * 32) measure_kernel(MeasureParams p) {
    __shared__ double res[kMeasBatch][6];  // chain: E, Y2, Y4, I; pair: q
    const int s = blockIdx.x / p.nT, t = blockIdx.x % p.nT, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SampleDev sd = p.samples[s];
    const int N = sd.N, R = p.R;
    const I per = (I)measure_tasks(R), total = (p.n_snap + (p.live ? 1 : 0)) * per;
    const int *perm = p.perm + (int64_t)s * R * p.nT;
    double *st = p.stat + ((int64_t)s * p.nT + t) * 7, *qs = p.qstat + ((int64_t)s * p.nT + t) * 5;
    unsigned long long *h = p.qhist + ((int64_t)s * p.nT + t) * 201;
    for (I b0 = 0; b0 < total; b0 += kMeasBatch) {
        const int n = (int)min((I)kMeasBatch, total - b0);
        for (int i = warp; i < n; i += kMeasWarps) {
            const int kk = (int)((b0 + i) / per);
            const I task = (b0 + i) - kk * per;
            const bool live = kk == p.n_snap;
            const V *a = live ? reinterpret_cast<const V *>(p.a) : reinterpret_cast<const V *>(p.snap_a) + (int64_t)kk * p.a_total;
            const double *E = live ? p.E : p.snap_E + (int64_t)kk * p.n_chains;
            if (task < R) {
                const int slot = perm[(int)task * p.nT + t];
                const V *x = a + sd.a_off + (int64_t)(slot - sd.chain0) * N;
                double i2 = 0.0, i4 = 0.0, i8 = 0.0;
                for (int k = lane; k < N; k += 32) {
                    const V v = x[k];
                    const double u = (double)v.x * v.x + (double)v.y * v.y;
                    i2 += u; i4 += u * u; i8 += (u * u) * (u * u);
                }
                for (int o = 16; o; o >>= 1) {
                    i2 += __shfl_xor_sync(0xffffffffu, i2, o);
                    i4 += __shfl_xor_sync(0xffffffffu, i4, o);
                    i8 += __shfl_xor_sync(0xffffffffu, i8, o);
                }
                if (lane == 0) { res[i][0] = E[slot]; res[i][1] = i4 / (i2 * i2); res[i][2] = i8 / (i4 * i4); res[i][3] = i2; }
            } else {
                int r1, r2;
                replica_pair(task - R, R, &r1, &r2);
                const V *x = a + sd.a_off + (int64_t)(perm[r1 * p.nT + t] - sd.chain0) * N;
                const V *y = a + sd.a_off + (int64_t)(perm[r2 * p.nT + t] - sd.chain0) * N;
                double d = 0.0;
                for (int k = lane; k < N; k += 32) {
                    const V u = x[k], v = y[k];
                    d += (double)u.x * v.x + (double)u.y * v.y;
                }
                for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                if (lane == 0) res[i][0] = d / (double)N;
            }
        }
        __syncthreads();
        const int w = threadIdx.x;
        if (w < 7) {  // n, E, E^2, Y2, Y4, I, I^2 over the chains of the batch
            double v = st[w];
            for (int i = 0; i < n; ++i) {
                if ((b0 + i) % per >= R) continue;
                const double e = res[i][0], i2 = res[i][3];
                v += w == 0 ? 1.0 : w == 1 ? e : w == 2 ? e * e : w == 3 ? res[i][1] : w == 4 ? res[i][2] : w == 5 ? i2 : i2 * i2;
            }
            st[w] = v;
        } else if (w >= 32 && w < 38) {  // n, q, q^2, q^3, q^4 and the histogram over the pairs
            const int m = w - 32;
            double v = m < 5 ? qs[m] : 0.0;
            for (int i = 0; i < n; ++i) {
                if ((b0 + i) % per < R) continue;
                const double q = res[i][0];
                if (m < 5) v += m == 0 ? 1.0 : m == 1 ? q : m == 2 ? q * q : m == 3 ? q * q * q : (q * q) * (q * q);
                else {
                    int b = (int)floor(100.0 * (q + 1.0) + 0.5);
                    b = b < 0 ? 0 : (b > 200 ? 200 : b);
                    h[b] += 1ull;
                }
            }
            if (m < 5) qs[m] = v;
        }
        __syncthreads();
    }
}

cudaError_t launch_measure(const MeasureParams &p, cudaStream_t s) {
    if (p.n_snap <= 0 && !p.live) return cudaSuccess;
    const int grid = p.S * p.nT;
    const bool wide = (p.n_snap + (p.live ? 1 : 0)) * measure_tasks(p.R) > (1 << 30);
    if (wide && p.dbl) measure_kernel<double2, int64_t><<<grid, kMeasWarps * 32, 0, s>>>(p);
    else if (wide) measure_kernel<float2, int64_t><<<grid, kMeasWarps * 32, 0, s>>>(p);
    else if (p.dbl) measure_kernel<double2, int><<<grid, kMeasWarps * 32, 0, s>>>(p);
    else measure_kernel<float2, int><<<grid, kMeasWarps * 32, 0, s>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// Plain FP64 path: the paper's GPU design restated (Sec. III.A.3): for every proposed pair move one
// thread per quadruplet holding j or k computes that quadruplet's energy change, the contributions are
// summed by a shared-memory tree reduction (O(log) depth), and one block simulates one chain; J is read
// from global memory by every chain separately.
__device__ __forceinline__ double2 cm(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double quad_term(double2 xa, double2 xb, double2 xc, double2 xd) {
    // Re( conj(a_a) a_b a_c conj(a_d) )
    const double2 ca = make_double2(xa.x, -xa.y), cd = make_double2(xd.x, -xd.y);
    return cm(cm(ca, xb), cm(xc, cd)).x;
}

__device__ __forceinline__ double tree_sum(double v, double *buf) {
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) buf[threadIdx.x] += buf[threadIdx.x + h];
        __syncthreads();
    }
    const double r = buf[0];
    __syncthreads();
    return r;
}

constexpr int kPlainThreads = 256;

__global__ void __launch_bounds__(kPlainThreads) plain_sweep_kernel(PlainParams p) {
    extern __shared__ double2 sa[];  // maxN amplitudes
    __shared__ double buf[kPlainThreads];
    __shared__ double2 s_new[2];
    __shared__ double s_U;
    const int slot = blockIdx.x;
    const int s = p.chain_sample[slot];
    const SampleDev sd = p.samples[s];
    const int N = sd.N, tid = threadIdx.x;
    const int r = (slot - sd.chain0) / p.nT, t = p.label[slot];
    const uint32_t cid = (uint32_t)((s * p.R + r) * p.nT + t);
    const double beta = p.beta[t];
    double2 *ag = p.a + sd.a_off + (int64_t)(slot - sd.chain0) * N;
    for (int k = tid; k < N; k += blockDim.x) sa[k] = ag[k];
    double E = p.E[slot];
    unsigned long long acc = 0, att = 0;
    const long long base = p.ctl->sweep_base;
    const int *inc_off = p.inc_off + sd.mode_off;
    const int *inc = p.inc + sd.inc_off;
    const int4 *quads = p.quads + sd.q_off;
    const double *Jq = p.Jq + sd.q_off;
    __syncthreads();
    for (int sw = 0; sw < p.n_sweeps; ++sw) {
        const uint32_t sweep = (uint32_t)(base + sw);
        for (int u = 0; u < N / 2; ++u) {
            int j, k;
            pair_jk(p.seed, (uint32_t)s, sweep, (uint32_t)u, N, j, k);
            if (tid == 0) {
                const u32x4 w = draw(p.seed, cid, sweep, (uint32_t)u, kTagPropose);
                const double2 aj = sa[j], ak = sa[k];
                const double uj = aj.x * aj.x + aj.y * aj.y, uk = ak.x * ak.x + ak.y * ak.y;
                const double K = sqrt(sqrt(uj * uj + uk * uk));
                const double phj = kTwoPi * u01(w.x), phk = kTwoPi * u01(w.y), th = kHalfPi * u01(w.z);
                const double Aj = K * sqrt(cos(th)), Ak = K * sqrt(sin(th));
                s_new[0] = make_double2(Aj * cos(phj), Aj * sin(phj));
                s_new[1] = make_double2(Ak * cos(phk), Ak * sin(phk));
                s_U = u01(w.w);
            }
            __syncthreads();
            const double2 nj = s_new[0], nk = s_new[1];
            const int oj = inc_off[j], nj_cnt = inc_off[j + 1] - oj;
            const int ok = inc_off[k], nk_cnt = inc_off[k + 1] - ok;
            double local = 0.0;
            for (int idx = tid; idx < nj_cnt + nk_cnt; idx += blockDim.x) {
                const int q = idx < nj_cnt ? inc[oj + idx] : inc[ok + idx - nj_cnt];
                const int4 Q = quads[q];
                const bool hasj = (Q.x == j || Q.y == j || Q.z == j || Q.w == j);
                if (idx >= nj_cnt && hasj) continue;  // counted once, from j's list
                double2 xa = sa[Q.x], xb = sa[Q.y], xc = sa[Q.z], xd = sa[Q.w];
                const double told = quad_term(xa, xb, xc, xd);
                if (Q.x == j) xa = nj; else if (Q.x == k) xa = nk;
                if (Q.y == j) xb = nj; else if (Q.y == k) xb = nk;
                if (Q.z == j) xc = nj; else if (Q.z == k) xc = nk;
                if (Q.w == j) xd = nj; else if (Q.w == k) xd = nk;
                local += Jq[q] * (quad_term(xa, xb, xc, xd) - told);
            }
            const double dH = -p.cc * tree_sum(local, buf);
            if (tid == 0) {
                ++att;
                if (dH <= 0.0 || s_U < exp(-beta * dH)) {
                    sa[j] = nj; sa[k] = nk;
                    E += dH;
                    ++acc;
                }
            }
            __syncthreads();
        }
        const long long done = base + sw + 1;
        if (p.measure_every > 0 && done % p.measure_every == 0 && sw + 1 < p.n_sweeps) {
            const int kk = (int)(done / p.measure_every - base / p.measure_every - 1);
            if (kk >= 0 && kk < p.n_snap_max) {
                double2 *dst = p.snap_a + (int64_t)kk * p.a_total + sd.a_off + (int64_t)(slot - sd.chain0) * N;
                for (int x = tid; x < N; x += blockDim.x) dst[x] = sa[x];
                if (tid == 0) p.snap_E[(int64_t)kk * p.n_chains + slot] = E;
            }
            __syncthreads();
        }
    }
    for (int x = tid; x < N; x += blockDim.x) ag[x] = sa[x];
    if (tid == 0) {
        p.E[slot] = E;
        p.mc_acc[slot] += acc;
        p.mc_att[slot] += att;
    }
}

__global__ void __launch_bounds__(kPlainThreads) plain_energy_kernel(PlainParams p) {
    extern __shared__ double2 sa[];
    __shared__ double buf[kPlainThreads];
    const int slot = blockIdx.x;
    const int s = p.chain_sample[slot];
    const SampleDev sd = p.samples[s];
    const int N = sd.N, tid = threadIdx.x;
    double2 *ag = p.a + sd.a_off + (int64_t)(slot - sd.chain0) * N;
    for (int k = tid; k < N; k += blockDim.x) sa[k] = ag[k];
    __syncthreads();
    if (p.renorm) {
        double s4 = 0.0;
        for (int k = tid; k < N; k += blockDim.x) {
            const double u = sa[k].x * sa[k].x + sa[k].y * sa[k].y;
            s4 += u * u;
        }
        s4 = tree_sum(s4, buf);
        if (!(s4 > 0.0) || !isfinite(s4)) record_error(p.ctl, kErrNaN, 20);
        const double f = sqrt(sqrt((double)N / s4));
        for (int k = tid; k < N; k += blockDim.x) {
            sa[k] = make_double2(sa[k].x * f, sa[k].y * f);
            ag[k] = sa[k];
        }
        __syncthreads();
    }
    const int4 *quads = p.quads + sd.q_off;
    const double *Jq = p.Jq + sd.q_off;
    const int64_t count = sd.nq;
    double local = 0.0;
    for (int64_t q = tid; q < count; q += blockDim.x) {
        const int4 Q = quads[q];
        local += Jq[q] * quad_term(sa[Q.x], sa[Q.y], sa[Q.z], sa[Q.w]);
    }
    const double E = -p.cc * tree_sum(local, buf);
    if (tid == 0) {
        if (!isfinite(E)) record_error(p.ctl, kErrNaN, 21);
        if (p.write_state) p.E[slot] = E;
        if (p.E_out) p.E_out[slot] = E;
    }
}

cudaError_t launch_plain_sweep(const PlainParams &p, int n_chains, cudaStream_t s) {
    if (n_chains <= 0 || p.n_sweeps <= 0) return cudaSuccess;
    plain_sweep_kernel<<<n_chains, kPlainThreads, (size_t)p.maxN * sizeof(double2), s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_plain_energy(const PlainParams &p, int n_chains, cudaStream_t s) {
    if (n_chains <= 0) return cudaSuccess;
    plain_energy_kernel<<<n_chains, kPlainThreads, (size_t)p.maxN * sizeof(double2), s>>>(p);
    return cudaGetLastError();
}

// Health check of the bounded waits: waits on a flag no kernel sets until the limit, then records the
// same timeout status as the engine's own waits.
__global__ void wait_probe_kernel(Control *ctl, unsigned long long limit_ns) {
    const volatile int *flag = &ctl->probe_flag;
    const unsigned long long t0 = global_ns();
    while (*flag == 0) {
        if (global_ns() - t0 > limit_ns) {
            record_error(ctl, kErrTimeout, 40);
            return;
        }
        __nanosleep(1000);
    }
}

cudaError_t launch_wait_probe(Control *ctl, unsigned long long limit_ns, cudaStream_t s) {
    wait_probe_kernel<<<1, 1, 0, s>>>(ctl, limit_ns);
    return cudaGetLastError();
}

__global__ void advance_kernel(Control *ctl, long long sweeps, long long passes, long long rounds) {
    ctl->sweep_base += sweeps;
    ctl->swap_passes += passes;
    ctl->global_rounds += rounds;
}

cudaError_t launch_advance(Control *ctl, long long sweeps, long long passes, long long rounds, cudaStream_t s) {
    advance_kernel<<<1, 1, 0, s>>>(ctl, sweeps, passes, rounds);
    return cudaGetLastError();
}

}  // namespace ptgb
