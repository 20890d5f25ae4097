// pt_row.cu -- one-chain-per-block Metropolis sweep on the comb graph (arXiv 2511.13508, Sec. III.A): the FP64
// sweep, and the FP32 sweep of small mode counts.
//
// The field of mode l factorises over the pair sum s = l + m (partner m):
//     h_l = sum_m conj(a_m) acc_l[m],   acc_l[m] = sum_{P = {x, s-x}} J_l[m][P] z_P,   z_P = a_x a_{s-x}.
// The chain's pair products z_P stay in shared memory for the whole launch; an accepted pair move rewrites the 2N - 3
// of them that hold j or k.  A thread evaluates one row (field j or k, partner m): two fused multiply-adds per
// coupling term, none for the product.
//
// Why one chain per block, without sharing J between chains: an SM does 2 FP64 fused multiply-adds per clock
// and 128 FP32 ones, so a warp's FP64 coupling term step (2 instructions, 32 clocks) hides a coalesced 256-byte
// coupling load from L1/L2 with ease, and forming the products again for every chain and update (as the J-sharing
// sweep does) would double the FP64 work.  Chains are the unit of scheduling, so that a small ensemble spreads over
// as many SMs as it has chains.
#include <cstdint>
#include "pt_common.cuh"
#include "pt_kernels.h"
#include "pt_move.cuh"

namespace ptgb {

namespace {

constexpr int kRowSmemMax = 227 * 1024;
constexpr int kRowDraws = 32;  // updates whose random numbers are drawn at once, one lane each
constexpr double kLeast = 4.9406564584124654e-324;  // the least positive double

// Pair products in rows by p, the pair's distance from the middle of its sum: pair {x, s-x}, x < s-x, is the p-th of
// sum s with p = (s-1)/2 - x.  Row p holds s = 2p+1 .. 2N-3-2p, so consecutive s (threads) are consecutive words, and
// the step from p to p+1 at the same s is 2N-5-4p.  N (N-1)/2 products, no gaps.
__host__ __device__ inline int pair_row(int p, int N) { return p * (2 * N - 3) - 2 * p * (p - 1) - (2 * p + 1); }
__device__ __forceinline__ int pair_index(int x, int s, int N) {
    const int p = ((s - 1) >> 1) - x;
    return pair_row(p, N) + s;
}
// pairs {x, y}, x < y, with x + y = s
__device__ __forceinline__ int pair_count(int s, int N) {
    return s < 1 ? 0 : ((s - 1) >> 1) - max(0, s - (N - 1)) + 1;
}

// The product of a pair, smaller mode first, with the fused multiply-adds written out: a launch forms it from the
// amplitudes, an accepted update again, and a run cut into launches has to round both alike.
template <typename V> __device__ __forceinline__ V pair_product(V lo, V hi) {
    V r;
    r.x = fma(lo.x, hi.x, -(lo.y * hi.y));
    r.y = fma(lo.x, hi.y, lo.y * hi.x);
    return r;
}

// A proposal as the rows use it.  test: FP32 the Metropolis uniform U; FP64 log U / (beta cc), drawn once with the proposal,
// so that the decision is one comparison: dH = -cc share, and U < exp(-beta dH) is share > log U / (beta cc), which holds for
// every dH <= 0 because log U < 0.  Where beta cc is infinite the quotient is -0; it is kept below zero, so that dH = 0 passes.
template <typename real> struct RowProposal {
    typename vec2<real>::type aj, ak, nj, nk, dj, dk;
    real test;
};
template <typename real> struct RowSmem {
    size_t a, draws, prop, part, pairs, total;
    __host__ __device__ RowSmem(int N) {
        using V = typename vec2<real>::type;
        a = (size_t)N * (N - 1) / 2 * sizeof(V);
        a = (a + 15) / 16 * 16;
        draws = a + (size_t)N * sizeof(V);
        draws = (draws + 15) / 16 * 16;
        prop = draws + 2 * kRowDraws * sizeof(ProposalDraw<real>);
        part = prop + 4 * sizeof(RowProposal<real>);
        pairs = part + 2 * 32 * sizeof(real);
        total = pairs + 2 * kRowDraws * sizeof(int);
    }
};

template <typename real> __device__ __forceinline__ bool row_accept(real share, real dH, real beta, real test) {
    if constexpr (sizeof(real) == 4) return metropolis_accept(dH, beta, test);
    else return share > test;
}

}  // namespace

// Threads: one per row (field j: partners 0..N-1, then field k), then one helper warp.  What the rows need but the
// state does not decide is kept off their path: the helper draws the random numbers of 32 updates at once (a lane
// each) half a batch ahead, and scales the proposal of the next update, for both outcomes of the current one.
// NP > 0 (rows of at most NP pairs): a row's couplings of the next update are loaded into registers while the current
// one is decided.
//
// dH = Re[conj(dj) h_j] with a_k already replaced + Re[conj(dk) h_k] with a_j not yet replaced (times -cc): the cross
// terms B_jk and A_jk then come from the one product and the one partner of a field-j row that hold k.
template <typename real, int NP, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) row_sweep_kernel(RowParams p) {
    using V = typename vec2<real>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    const RowSmem<real> lay(p.maxN);
    V *z = reinterpret_cast<V *>(smem);
    V *a = reinterpret_cast<V *>(smem + lay.a);
    ProposalDraw<real> *draws = reinterpret_cast<ProposalDraw<real> *>(smem + lay.draws);  // [2][kRowDraws]
    RowProposal<real> *prop = reinterpret_cast<RowProposal<real> *>(smem + lay.prop);      // [2][2]
    real *part = reinterpret_cast<real *>(smem + lay.part);                                // [2][32]
    int *pairs = reinterpret_cast<int *>(smem + lay.pairs);                                // [2][kRowDraws]

    const int slot = p.order[blockIdx.x];
    const int si = p.chain_sample[slot];
    const SampleDev sd = p.samples[si];
    const int N = sd.N, half = N / 2, tid = threadIdx.x, T = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const int RW = (T >> 5) - 1;  // row warps
    const bool helper = warp == RW;
    const int r = (slot - sd.chain0) / p.nT, t = p.label[slot];
    const uint32_t cid = (uint32_t)((si * p.R + r) * p.nT + t);
    const real beta = (real)p.beta[t], cc = (real)p.cc;
    V *ag = reinterpret_cast<V *>(p.a) + sd.a_off + (int64_t)(slot - sd.chain0) * N;
    const real *J = reinterpret_cast<const real *>(p.J) + sd.row_off;
    const long long base = p.ctl->sweep_base;
    const long long tr_at = p.trace ? p.ctl->trace_at : 0ll;
    const int tr_u = p.trace ? p.ctl->trace_update : -1;
    const int total = p.n_sweeps * half;

    // random numbers of updates [n0, n0 + kRowDraws): lane l's update goes to slot (n0 + l) of the two-batch ring
    auto draw_batch = [&](int n0) {
        const int n = n0 + lane;
        if (n < total) {
            const int sw = n / half, u = n - sw * half, at = n & (2 * kRowDraws - 1);
            int j, k;
            pair_jk(p.seed, (uint32_t)si, (uint32_t)(base + sw), (uint32_t)u, N, j, k);
            pairs[at] = j | (k << 16);
            ProposalDraw<real> D = draw_proposal<real>(p.seed, cid, (uint32_t)(base + sw), (uint32_t)u);
            if constexpr (sizeof(real) == 8) { D.pad = D.U; D.U = fmin(log(D.U) / (beta * cc), -kLeast); }
            draws[at] = D;
        }
    };
    for (int x = tid; x < N; x += T) a[x] = ag[x];
    if (helper) draw_batch(0);
    __syncthreads();
    for (int y = 1; y < N; ++y)
        for (int x = tid; x < y; x += T) z[pair_index(x, x + y, N)] = pair_product(a[x], a[y]);
    double E = p.E[slot];
    unsigned long long acc_n = 0;

    // this thread's row: partner m of field j or k
    const bool fk = tid >= N;
    const int m = fk ? tid - N : tid;
    const bool has_row = !helper && m < N;
    int n = 0, s = 0, y = -1;      // pairs in the row, pair sum, partner of k in the row's pair that holds k (-1: none)
    const real *Jr = J;
    real Jreg[NP > 0 ? NP : 1], Jb = real(0);
    auto row_of = [&](int jk) {
        const int j = jk & 0xffff, k = jk >> 16, l = fk ? k : j;
        s = l + m;
        n = (has_row && m != l) ? pair_count(s, N) : 0;
        Jr = J + l * half * N + m;
        y = s - k;
        if (fk || n <= 0 || y < 0 || y >= N || y == k) y = -1;
        Jb = y >= 0 ? __ldg(Jr + (((s - 1) >> 1) - min(k, y)) * N) : real(0);
        if constexpr (NP > 0) {
#pragma unroll
            for (int e = 0; e < NP; ++e) Jreg[e] = e < n ? __ldg(Jr + e * N) : real(0);
        }
    };
    if (has_row && total > 0) row_of(pairs[0]);
    auto propose = [&](RowProposal<real> &o, const ProposalDraw<real> &D, V aj, V ak) {
        const Proposal<real> P = finish_proposal<real>(D, aj, ak);
        o.aj = aj; o.ak = ak; o.nj = P.nj; o.nk = P.nk; o.test = P.U;
        o.dj.x = P.nj.x - aj.x; o.dj.y = P.nj.y - aj.y;
        o.dk.x = P.nk.x - ak.x; o.dk.y = P.nk.y - ak.y;
    };
    if (helper && lane < 2 && total > 0) {
        const int jk = pairs[0];
        propose(prop[lane], draws[0], a[jk & 0xffff], a[jk >> 16]);
    }
    __syncthreads();

    int ok = 0, at_u = 0, sw = 0;
    for (int i = 0; i < total; ++i) {
        const int jk = pairs[i & (2 * kRowDraws - 1)], j = jk & 0xffff, k = jk >> 16;
        const RowProposal<real> &P = prop[(i & 1) * 2 + ok];
        const bool traced = tr_at == base + sw + 1 && at_u == tr_u;
        real share = 0;
        V acc;
        acc.x = acc.y = real(0);
        if (has_row) {
            V ac2;
            ac2.x = ac2.y = real(0);
            int zi = s - 1, step = 2 * N - 5;
            if constexpr (NP > 0) {
                // past the row's end the coupling is zero and the product any one: no branches
#pragma unroll
                for (int e = 0; e < NP; ++e) {
                    caxpy((e & 1) ? ac2 : acc, Jreg[e], z[e < n ? zi : 0]);
                    zi += step; step -= 4;
                }
            } else {
                int e0 = 0;
                for (; e0 + 8 <= n; e0 += 8) {
                    real Jv[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) Jv[e] = __ldg(Jr + (e0 + e) * N);
#pragma unroll
                    for (int e = 0; e < 8; ++e) { caxpy((e & 1) ? ac2 : acc, Jv[e], z[zi]); zi += step; step -= 4; }
                }
                if (e0 < n) {
                    real Jv[8];
#pragma unroll
                    for (int e = 0; e < 7; ++e) Jv[e] = e0 + e < n ? __ldg(Jr + (e0 + e) * N) : real(0);
#pragma unroll
                    for (int e = 0; e < 7; ++e)
                        if (e0 + e < n) { caxpy((e & 1) ? ac2 : acc, Jv[e], z[zi]); zi += step; step -= 4; }
                }
            }
            acc.x += ac2.x; acc.y += ac2.y;
            // share = Re[conj(d) conj(a_m) x] = Re[conj(d a_m) x], x = acc, for field j with a_k replaced: the pair {k, y}
            // changes by dk a_y, and partner k is nk.  d a_m and J a_y wait for no sum
            const V d = fk ? P.dk : P.dj, am = (!fk && m == k) ? P.nk : a[m], dm = cmul(d, am);
            V x = acc;
            const V ay = a[y >= 0 ? y : 0], dk = P.dk;
            const real tx = Jb * ay.x, ty = Jb * ay.y;  // zero coupling where there is no such pair
            x.x = fma(dk.x, tx, fma(-dk.y, ty, x.x));
            x.y = fma(dk.x, ty, fma(dk.y, tx, x.y));
            share = fma(dm.x, x.x, dm.y * x.y);
        }
        if (!helper) {
#pragma unroll
            for (int o = 16; o; o >>= 1) share += __shfl_xor_sync(0xffffffffu, share, o);
            if (lane == 0) part[(i & 1) * 32 + warp] = share;
        } else {
            if ((i & (kRowDraws - 1)) == kRowDraws / 2) draw_batch((i & ~(kRowDraws - 1)) + kRowDraws);
            __syncwarp();
            if (lane < 2 && i + 1 < total) {  // the next update's proposal if this one is rejected (lane 0) or accepted
                const int at = (i + 1) & (2 * kRowDraws - 1), nx = pairs[at], j2 = nx & 0xffff, k2 = nx >> 16;
                V aj = a[j2], ak = a[k2];
                if (lane == 1) {
                    if (j2 == j) aj = P.nj; else if (j2 == k) aj = P.nk;
                    if (k2 == j) ak = P.nj; else if (k2 == k) ak = P.nk;
                }
                propose(prop[((i + 1) & 1) * 2 + lane], draws[at], aj, ak);
            }
        }
        if (traced) {  // the record of this update (h_j, h_k, B_jk, A_jk) and the state before it
            V v[4];
            for (int e = 0; e < 4; ++e) v[e].x = v[e].y = real(0);
            if (has_row) {
                v[fk ? 1 : 0] = cmulc(a[m], acc);
                if (y >= 0) { v[2] = cmulc(a[m], a[y]); v[2].x *= Jb; v[2].y *= Jb; }
                if (!fk && m == k) v[3] = acc;
            }
            double *rec = p.trace + (int64_t)cid * kTraceRec;
            for (int e = 0; e < 4; ++e) {
                real vx = v[e].x, vy = v[e].y;
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    vx += __shfl_xor_sync(0xffffffffu, vx, o);
                    vy += __shfl_xor_sync(0xffffffffu, vy, o);
                }
                real *px = part + ((i + 1) & 1) * 32;
                if (lane == 0) { px[2 * warp] = vx; px[2 * warp + 1] = vy; }
                __syncthreads();
                if (tid == 0) {
                    double hx = 0, hy = 0;
                    for (int w = 0; w < RW; ++w) { hx += (double)px[2 * w]; hy += (double)px[2 * w + 1]; }
                    rec[2 + 2 * e] = hx; rec[3 + 2 * e] = hy;
                }
                __syncthreads();
            }
            double2 *st = reinterpret_cast<double2 *>(p.trace + (int64_t)p.n_chains * kTraceRec) + sd.a_off +
                          (int64_t)(cid - (uint32_t)sd.chain0) * N;
            for (int x = tid; x < N; x += T) st[x] = make_double2((double)a[x].x, (double)a[x].y);
        }
        __syncthreads();
        share = part[(i & 1) * 32];
        for (int w = 1; w < RW; ++w) share += part[(i & 1) * 32 + w];
        const real dH = -cc * share;
        const bool take = row_accept<real>(share, dH, beta, P.test);
        if (traced && tid == 0) {
            const ProposalDraw<real> &D = draws[i & (2 * kRowDraws - 1)];
            double *rec = p.trace + (int64_t)cid * kTraceRec;
            rec[0] = j; rec[1] = k;
            rec[10] = P.nj.x; rec[11] = P.nj.y; rec[12] = P.nk.x; rec[13] = P.nk.y;
            rec[14] = sizeof(real) == 8 ? D.pad : D.U;
            rec[15] = dH; rec[16] = take ? 1.0 : 0.0; rec[17] = beta; rec[18] = E; rec[19] = 1.0;
        }
        if (take) {
            if (tid == 0) { E += (double)dH; ++acc_n; }
            // the products that hold j or k; always smaller mode times larger, as at the start of a launch
            const int l = fk ? k : j;
            if (has_row && m != l && !(fk && m == j)) {
                const V nl = fk ? P.nk : P.nj, nm = (!fk && m == k) ? P.nk : a[m];
                z[pair_index(min(l, m), l + m, N)] = l < m ? pair_product(nl, nm) : pair_product(nm, nl);
            }
            if (helper && lane == 0) { a[j] = P.nj; a[k] = P.nk; }
        }
        if (has_row && i + 1 < total) row_of(pairs[(i + 1) & (2 * kRowDraws - 1)]);
        ok = take ? 1 : 0;
        __syncthreads();
        if (++at_u == half) {
            at_u = 0; ++sw;
            const long long done = base + sw;
            if (p.measure_every > 0 && done % p.measure_every == 0 && sw < p.n_sweeps) {
                const int kk = (int)(done / p.measure_every - base / p.measure_every - 1);
                if (kk >= 0 && kk < p.n_snap_max) {
                    V *dst = reinterpret_cast<V *>(p.snap_a) + (int64_t)kk * p.a_total + sd.a_off +
                             (int64_t)(slot - sd.chain0) * N;
                    for (int x = tid; x < N; x += T) dst[x] = a[x];
                    if (tid == 0) p.snap_E[(int64_t)kk * p.n_chains + slot] = E;
                }
            }
        }
    }
    for (int x = tid; x < N; x += T) ag[x] = a[x];
    if (tid == 0) {
        p.E[slot] = E;
        p.mc_acc[slot] += acc_n;
        p.mc_att[slot] += (unsigned long long)total;
    }
}

// Couplings by (mode, pair distance p, partner m): J_l[p][m], zero where {l, m} and the p-th pair of sum l + m
// do not make a quadruplet.  One thread per quadruplet {a, d} u {b, c}, a + d = b + c: it belongs to four rows.
template <typename real>
__global__ void row_pack_kernel(const SampleDev *samples, const int4 *quads, const double *Jq, real *out) {
    const SampleDev sd = samples[blockIdx.y];
    const int N = sd.N, half = N / 2;
    real *J = out + sd.row_off;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < sd.nq; q += (int64_t)gridDim.x * blockDim.x) {
        const int4 Q = quads[sd.q_off + q];
        const real v = (real)Jq[sd.q_off + q];
        const int mid = (Q.x + Q.w - 1) >> 1;
        const size_t pa = (size_t)(mid - Q.x) * N, pb = (size_t)(mid - Q.y) * N;
        J[(size_t)Q.x * half * N + pb + Q.w] = v;
        J[(size_t)Q.w * half * N + pb + Q.x] = v;
        J[(size_t)Q.y * half * N + pa + Q.z] = v;
        J[(size_t)Q.z * half * N + pa + Q.y] = v;
    }
}

cudaError_t launch_row_pack(bool dbl, const SampleDev *samples, int S, const int4 *quads, const double *Jq, void *out,
                            cudaStream_t s) {
    const dim3 grid(32, S);
    if (dbl) row_pack_kernel<double><<<grid, 256, 0, s>>>(samples, quads, Jq, reinterpret_cast<double *>(out));
    else row_pack_kernel<float><<<grid, 256, 0, s>>>(samples, quads, Jq, reinterpret_cast<float *>(out));
    return cudaGetLastError();
}

size_t row_smem_bytes(bool dbl, int maxN) { return dbl ? RowSmem<double>(maxN).total : RowSmem<float>(maxN).total; }

// GB300, us per sweep: N = 16, 64 chains FP64 16.7 (268 on J-sharing blocks of 16 chains, 4 SMs busy); N = 64, 1024 chains
// FP64 856 (2230 on blocks of 8, 4187 of 16), 4096 chains 3460 (6110); N = 128, 512 chains FP64 2990 (10270); N = 18, 168
// chains FP32 8.0 (17.1); N = 32, 168 chains FP32 14.3 (32).  What is left of an update of few rows is a chain of FP64
// latencies (about 70 clocks each); a third warp for the random numbers alone gained 5% there and cost as much at FP32.
// Variants by the largest N: rows of at most 8 or 16 pairs keep their couplings in registers; longer rows load them in
// eights.  The register budget follows the blocks an SM holds at that N (pair products of 227 KB).  FP32 rows end at N = 48.
#define PT_ROW_DISPATCH(T, CALL)                                                                      \
    constexpr bool kF = sizeof(T) == 4;                                                               \
    if (maxN <= 16) { auto *k = row_sweep_kernel<T, 8, 64, kF ? 8 : 10>; CALL; }                     \
    else if (maxN <= 32) { auto *k = row_sweep_kernel<T, 16, 96, kF ? 7 : 6>; CALL; }                 \
    else if (maxN <= 64) { auto *k = row_sweep_kernel<T, 0, 160, kF ? 5 : 6>; CALL; }                 \
    else { auto *k = row_sweep_kernel<T, 0, kF ? 160 : kRowMaxThreads, kF ? 5 : 1>; CALL; }

// The limit is the kernel's largest (kRowSmemMax), not this context's: contexts of other sizes launch the same kernel.
cudaError_t row_prepare(bool dbl, int maxN) {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (dbl) { PT_ROW_DISPATCH(double, return cudaFuncSetAttribute(k, at, kRowSmemMax)) }
    else { PT_ROW_DISPATCH(float, return cudaFuncSetAttribute(k, at, kRowSmemMax)) }
}

cudaError_t launch_row_sweep(bool dbl, const RowParams &p, cudaStream_t s) {
    if (p.n_chains <= 0 || p.n_sweeps <= 0) return cudaSuccess;
    const int maxN = p.maxN, threads = ((2 * maxN + 31) / 32 + 1) * 32;
    const size_t sm = row_smem_bytes(dbl, maxN);
    if (dbl) { PT_ROW_DISPATCH(double, (k<<<p.n_chains, threads, sm, s>>>(p))) }
    else { PT_ROW_DISPATCH(float, (k<<<p.n_chains, threads, sm, s>>>(p))) }
    return cudaGetLastError();
}

}  // namespace ptgb
