// pt_sweep.cu -- the J-sharing FP64 Metropolis sweep kernel (sm_103a), the field-only kernel and the
// full-energy (resync) kernel, for the smoothed-cubic 4-body random-laser model (arXiv 2511.13508).
//
// Local field of the updated modes (paper Sec. III.A.3).  With z_P = a_x a_y for the pair P = {x,y},
// the field of mode l factorises over the pair sum s = x + y:
//     h_l = sum_s conj(a_{s-l}) acc_l[s],     acc_l[s] = sum_{P : x+y=s} J_l[s][P] z_P,
// where J_l[s][P] is the coupling of quadruplet {l, s-l} u P.  One pair product z_P therefore feeds
// both fields of a pair update (j,k), and all chains of a disorder sample read J_j and J_k once per
// thread block: the J rows stream HBM/L2 -> shared memory through cp.async.bulk (TMA) into a ring of
// stages, guarded by mbarriers, while the chains' amplitudes stay resident in shared memory.
//
// Delta H of a pair move (j,k) (Sec. III.A.1; cross term = reading R5 of the design notes):
//     dH = -cc Re[ conj(dj) h_j + conj(dk) h_k + conj(dj) dk B_jk + conj(dj) conj(dk) A_jk ],
//     B_jk = sum_s conj(a_{s-j}) J_j[s][{k, s-k}] a_{s-k},   A_jk = acc_j[j+k].
#include <cstdint>
#include <cstdio>
#include "pt_bulk.cuh"
#include "pt_common.cuh"
#include "pt_kernels.h"
#include "pt_rules.h"
#include "pt_move.cuh"

namespace ptgb {

// Row-stride of the shared amplitude table [x + APAD][chain] (complex elements): one pad element for
// 8-byte complex with 8 chains, so that four workers reading rows 8 apart hit distinct bank halves.
template <typename real, int G> struct RowStride {
    static constexpr int value = (sizeof(real) == 4 && G == 8) ? G + 1 : G;
};

// Loads one J column (TS reals: fixed x offset, the TS rows) of a block as vectors.
template <typename real> struct JRow;
template <> struct JRow<float> {
    float v[TX];
    __device__ __forceinline__ void load(const float *p) {
        const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
};
template <> struct JRow<double> {
    double v[TX];
    __device__ __forceinline__ void load(const double *p) {
#pragma unroll
        for (int i = 0; i < TX; i += 2) {
            const double2 a = *reinterpret_cast<const double2 *>(p + i);
            v[i] = a.x; v[i + 1] = a.y;
        }
    }
};

// Per-lane partial sums of one pair update.
template <typename real> struct Partials {
    typename vec2<real>::type hj, hk, B, A;
    __device__ __forceinline__ void zero() {
        hj.x = hj.y = hk.x = hk.y = B.x = B.y = A.x = A.y = real(0);
    }
};

// h += conj(m) acc, as four fused multiply-adds
template <typename V> __device__ __forceinline__ void cfma_conj(V &h, V m, V acc) {
    h.x = fma(m.x, acc.x, h.x);
    h.x = fma(m.y, acc.y, h.x);
    h.y = fma(m.x, acc.y, h.y);
    h.y = fma(-m.y, acc.x, h.y);
}

// One TS x TX block of pair products for chain c: accumulates the j field (MODE & 1), the k field
// (MODE & 2), and the j-k cross terms (with the j field).  as = shared amplitude table; Jj, Jk =
// column-major blocks.  The x offset i runs outside, the row r inside, so the 2*TS row accumulators
// are independent chains of fused multiply-adds.
template <typename real, int RS, int MODE, bool WB>
__device__ __forceinline__ void process_block(const typename vec2<real>::type *__restrict__ as, int c, int s0,
                                              int x0, int j, int k, int N, const real *Jj, const real *Jk,
                                              Partials<real> &p) {
    using V = typename vec2<real>::type;
    V ax[TX], ay[TS + TX - 1];
#pragma unroll
    for (int i = 0; i < TX; ++i) ax[i] = as[(x0 + i + APAD) * RS + c];
    const int ybase = s0 - x0 - (TX - 1) + APAD;
#pragma unroll
    for (int d = 0; d < TS + TX - 1; ++d) ay[d] = as[(ybase + d) * RS + c];
    V accj[TS], acck[TS];
#pragma unroll
    for (int r = 0; r < TS; ++r) accj[r].x = accj[r].y = acck[r].x = acck[r].y = real(0);
#pragma unroll
    for (int i = 0; i < TX; ++i) {
        JRow<real> cj, ck;
        if (MODE & 1) cj.load(Jj + i * TS);
        if (MODE & 2) ck.load(Jk + i * TS);
#pragma unroll
        for (int r = 0; r < TS; ++r) {
            const V z = cmul(ax[i], ay[r - i + TX - 1]);
            if (MODE & 1) caxpy(accj[r], cj.v[r], z);
            if (MODE & 2) caxpy(acck[r], ck.v[r], z);
        }
    }
#pragma unroll
    for (int r = 0; r < TS; ++r) {
        const int s = s0 + r;
        if (MODE & 1) cfma_conj(p.hj, as[(s - j + APAD) * RS + c], accj[r]);
        if (MODE & 2) cfma_conj(p.hk, as[(s - k + APAD) * RS + c], acck[r]);
    }
    if (MODE & 1) {
        // A_jk is the accumulator of row j+k: only the blocks of that row's s-tile hold it
        const int rs = j + k - s0;
        if (rs >= 0 && rs < TS) {
#pragma unroll
            for (int r = 0; r < TS; ++r)
                if (r == rs) cadd(p.A, accj[r]);
        }
    }
    if ((MODE & 1) && WB) {
        // B_jk: the element of row s at x* = min(k, s-k) belongs to this block for the rows s >= 2k of
        // the column tile holding k, and for the rows s - k in [x0, x0+TX) of the diagonal band.
        const bool col = (k >= x0 && k < x0 + TX);
        const bool diag = (s0 + TS - 1 >= x0 + k) && (s0 <= x0 + TX - 1 + k);
        if (col || diag) {
#pragma unroll
            for (int r = 0; r < TS; ++r) {
                const int s = s0 + r, y = s - k;
                const int xs = (y < k) ? y : k;
                if (y >= 0 && y < N && xs >= x0 && xs < x0 + TX) {
                    const real Jv = Jj[(xs - x0) * TS + r];
                    const V m = as[(s - j + APAD) * RS + c];
                    const V yv = as[(y + APAD) * RS + c];
                    caxpy(p.B, Jv, cmulc(m, yv));
                }
            }
        }
    }
}

template <typename real, int RS, bool WB>
__device__ __forceinline__ void process_block_dispatch(int mode, const typename vec2<real>::type *as, int c,
                                                       int s0, int x0, int j, int k, int N, const real *Jj,
                                                       const real *Jk, Partials<real> &p) {
    if (mode == 3) process_block<real, RS, 3, WB>(as, c, s0, x0, j, k, N, Jj, Jk, p);
    else if (mode == 1) process_block<real, RS, 1, WB>(as, c, s0, x0, j, k, N, Jj, Jk, p);
    else if (mode == 2) process_block<real, RS, 2, WB>(as, c, s0, x0, j, k, N, Jj, Jk, p);
}


// Block ranges of an update: union of the runs of j and k in the sample's block list.
struct Ranges {
    int jlo, jhi, klo, khi, ulo, uhi;  // sample-local block indices [lo, hi)
    int64_t jg, kg;                    // global block index of the first block of j's / k's run
};
__device__ __forceinline__ Ranges update_ranges(const SampleDev &sd, const int *bo, const int *mode_blk, int j,
                                                int k) {
    Ranges R;
    const int stlo_j = j / TS, sthi_j = min((j + sd.N - 1) / TS, sd.ST - 1);
    const int stlo_k = k / TS, sthi_k = min((k + sd.N - 1) / TS, sd.ST - 1);
    R.jlo = bo[stlo_j]; R.jhi = bo[sthi_j + 1];
    R.klo = bo[stlo_k]; R.khi = bo[sthi_k + 1];
    R.ulo = min(R.jlo, R.klo); R.uhi = max(R.jhi, R.khi);
    R.jg = sd.J_off + mode_blk[j];
    R.kg = sd.J_off + mode_blk[k];
    return R;
}

// With 8 chains per block the copy warp also draws the random part of every chain's proposal, up to kBD updates ahead,
// and warp 0 only finishes it at the update's start; with 16 chains warp 0 draws the whole proposal itself.
template <int G> constexpr bool kCopyDraws = G == 8;

template <typename real>
__device__ __forceinline__ real delta_h(const Proposal<real> &P, const Partials<real> &f, real cc) {
    using V = typename vec2<real>::type;
    V dj, dk;
    dj.x = P.nj.x - P.aj.x; dj.y = P.nj.y - P.aj.y;
    dk.x = P.nk.x - P.ak.x; dk.y = P.nk.y - P.ak.y;
    const V t1 = cmulc(dj, f.hj), t2 = cmulc(dk, f.hk);
    const V djdk = cmulc(dj, dk);  // conj(dj) dk
    V cdjcdk;                      // conj(dj) conj(dk)
    cdjcdk.x = dj.x * dk.x - dj.y * dk.y;
    cdjcdk.y = -(dj.x * dk.y + dj.y * dk.x);
    const V t3 = cmul(djdk, f.B), t4 = cmul(cdjcdk, f.A);
    return -cc * (t1.x + t2.x + t3.x + t4.x);
}

// Update trace: one chain's record of the traced update and its state before the update (modes j and k from
// the proposal's old amplitudes: the other warps may already have written the new ones).
template <typename real, int RS>
__device__ __noinline__ void trace_write(double *trace, int n_chains, int64_t a_off, int chain0, int N, uint32_t id,
                                         int j, int k, Partials<real> f, Proposal<real> P, real dH, bool acc,
                                         real beta, double E, const typename vec2<real>::type *as, int c) {
    using V = typename vec2<real>::type;
    double *rec = trace + (int64_t)id * kTraceRec;
    const double v[kTraceRec] = {(double)j, (double)k, (double)f.hj.x, (double)f.hj.y, (double)f.hk.x,
                                 (double)f.hk.y, (double)f.B.x, (double)f.B.y, (double)f.A.x, (double)f.A.y,
                                 (double)P.nj.x, (double)P.nj.y, (double)P.nk.x, (double)P.nk.y, (double)P.U,
                                 (double)dH, acc ? 1.0 : 0.0, (double)beta, E, 1.0};
    for (int e = 0; e < kTraceRec; ++e) rec[e] = v[e];
    double2 *st = reinterpret_cast<double2 *>(trace + (int64_t)n_chains * kTraceRec) + a_off +
                  (int64_t)(id - (uint32_t)chain0) * N;
    for (int x = 0; x < N; ++x) {
        const V a = (x == j) ? P.aj : (x == k) ? P.ak : as[(x + APAD) * RS + c];
        st[x] = make_double2((double)a.x, (double)a.y);
    }
}

// ------------------------------------------------------------------------------------------------
// The persistent FP64 sweep kernel of explicit block shapes and of N > 160 (the others run one chain per block,
// pt_row.cu; FP32: pt_comb.cu).  NCW consumer warps + 1 producer warp.  A consumer lane is
// (chain c = lane % G, worker q = lane / G); worker w = warp * (32/G) + q takes block w of every
// chunk of CB = NCW*32/G blocks.  The producer (copy) warp streams the J runs of j and k, chunk by chunk,
// into a ring of NST stages and, with 8 chains per block, draws the random part of every chain's proposal into one
// slot per update of a second ring (kBD slots).  Work units = (group, run of sweeps) come from a ticket counter; a unit
// waits (bounded) until the previous run of its group has been written back.
// Ring depth: as many stages as fit next to the amplitude table of the largest N (up to kNstMax), so
// that the copies of a chunk are issued several chunks ahead of its use (L2 misses of the coupling runs).
constexpr int kNstMax = 6, kNstMin = 2;
// Proposal slots: the copy warp is up to kBD updates ahead of the field warps.
constexpr int kBD = 4;

template <typename real, int G, int NCW> struct SweepShape {
    static constexpr int WPW = 32 / G;
    static constexpr int NW = NCW * WPW;
    static constexpr int CB = NW;
    static constexpr int RS = RowStride<real, G>::value;
    static constexpr int NTHREADS = (NCW + 1) * 32;
    static constexpr int JS = JStride<real>::value;
    static constexpr size_t stage_bytes = (size_t)2 * CB * JS * sizeof(real);
};

// Shared memory of the sweep kernel without the coupling ring.
template <typename real, int G, int NCW> size_t sweep_fixed_bytes(int maxN) {
    using Sh = SweepShape<real, G, NCW>;
    using V = typename vec2<real>::type;
    size_t b = 0;
    b += 2 * (kNstMax + kBD) * sizeof(uint64_t);                          // mbarriers
    b = (b + 127) / 128 * 128;
    b += (size_t)(maxN + 2 * APAD) * Sh::RS * sizeof(V);                  // amplitudes
    b += (size_t)2 * NCW * G * 8 * sizeof(real);                          // reduction, double-buffered
    if (kCopyDraws<G>) b += (size_t)kBD * G * sizeof(ProposalDraw<real>);  // proposal draws of kBD updates
    b += (size_t)2 * G * sizeof(Proposal<real>) + 16;                     // proposals, double-buffered
    b += (size_t)G * (sizeof(double) + sizeof(real) + 2 * sizeof(uint32_t) + sizeof(unsigned long long));
    b += (size_t)(2 * 128 + 8) * sizeof(int);                             // bo / xtlo tables
    b += (size_t)(maxN / 2) * sizeof(int);                                // pair sequence of a sweep
    b += 64;
    return b;
}

// Ring stages for the largest N within `limit` bytes of shared memory per block (0 when fewer than kNstMin fit).
template <typename real, int G, int NCW> int sweep_stages(int maxN, size_t limit) {
    const size_t fixed = sweep_fixed_bytes<real, G, NCW>(maxN), st = SweepShape<real, G, NCW>::stage_bytes;
    if (fixed + kNstMin * st > limit) return 0;
    const size_t n = (limit - fixed) / st;
    return n > (size_t)kNstMax ? kNstMax : (int)n;
}

template <typename real, int G, int NCW> size_t sweep_smem_bytes(int maxN, int nst) {
    return sweep_fixed_bytes<real, G, NCW>(maxN) + (size_t)nst * SweepShape<real, G, NCW>::stage_bytes;
}

template <typename real, int G, int NCW>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) sweep_kernel(SweepParams prm) {
    using Sh = SweepShape<real, G, NCW>;
    using V = typename vec2<real>::type;
    constexpr int RS = Sh::RS, CB = Sh::CB, WPW = Sh::WPW, JS = Sh::JS;
    const int NST = prm.nst;  // ring stages (kNstMin .. kNstMax), chosen by the launcher for the largest N
    constexpr int NCT = NCW * 32;  // consumer threads
    // decision step (see the end of an update): 16 chains per block spread it over 8 lanes per chain, 8 chains take it
    // redundantly in every warp
    constexpr bool kSpread = G == 16;

    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);
    uint64_t *empty = full + kNstMax;
    uint64_t *bfull = empty + kNstMax;  // B-coupling buffers: filled (32 copy-warp lanes) / read (NCW warps)
    uint64_t *bempty = bfull + kBD;
    size_t off = (2 * (kNstMax + kBD) * sizeof(uint64_t) + 127) / 128 * 128;
    real *ring = reinterpret_cast<real *>(smem + off);
    off += NST * Sh::stage_bytes;
    V *as = reinterpret_cast<V *>(smem + off);
    off += (size_t)(prm.maxN + 2 * APAD) * RS * sizeof(V);
    real *red = reinterpret_cast<real *>(smem + off);
    off += (size_t)2 * NCW * G * 8 * sizeof(real);
    off = (off + 15) / 16 * 16;
    ProposalDraw<real> *pdraw = nullptr;  // [kBD][G]
    if (kCopyDraws<G>) {
        pdraw = reinterpret_cast<ProposalDraw<real> *>(smem + off);
        off += (size_t)kBD * G * sizeof(ProposalDraw<real>);
    }
    Proposal<real> *prop = reinterpret_cast<Proposal<real> *>(smem + off);
    off += (size_t)2 * G * sizeof(Proposal<real>);
    double *cE = reinterpret_cast<double *>(smem + off);
    off += G * sizeof(double);
    real *cBeta = reinterpret_cast<real *>(smem + off);
    off += G * sizeof(real);
    uint32_t *cId = reinterpret_cast<uint32_t *>(smem + off);
    off += G * sizeof(uint32_t);
    uint32_t *cAcc = reinterpret_cast<uint32_t *>(smem + off);
    off += G * sizeof(uint32_t);
    off = (off + 7) / 8 * 8;
    unsigned long long *cAtt = reinterpret_cast<unsigned long long *>(smem + off);
    off += G * sizeof(unsigned long long);
    int *s_bo = reinterpret_cast<int *>(smem + off);
    off += 129 * sizeof(int);
    int *s_xtlo = reinterpret_cast<int *>(smem + off);
    off += 129 * sizeof(int);
    int *s_unit = reinterpret_cast<int *>(smem + off);  // [0] group, [1] chunk, [2] abort
    volatile int *abort_flag = s_unit + 2;
    int *s_pair = s_unit + 4;  // (j | k << 16) of every update of the current sweep

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const bool producer = (warp == NCW);
    const int c = lane % G, wq = lane / G;
    // warp 0 also draws the proposals, so it takes the last workers of a chunk: it is the one left without a
    // block when an update's last chunk is not full
    const int worker = (warp == 0 ? NCW - 1 : warp - 1) * WPW + wq;

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NCW);
        }
        for (int i = 0; i < kBD; ++i) {
            mbar_init(&bfull[i], 32);
            mbar_init(&bempty[i], NCW);
        }
        s_unit[2] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();

    const long long sweep_base = prm.ctl->sweep_base;
    const int n_sweeps = prm.n_sweeps, spu = prm.sweeps_per_unit;
    const int chunks_per_group = (n_sweeps + spu - 1) / spu;
    const unsigned total_units = (unsigned)chunks_per_group * (unsigned)prm.n_groups;
    const real *J = reinterpret_cast<const real *>(prm.J);
    V *A = reinterpret_cast<V *>(prm.a);
    uint32_t q = 0;  // global chunk counter (ring position)
    // ring stage of chunk q (q mod NST) and the parity of its pass through the ring, advanced with q (NST is a
    // launch parameter: no division per chunk)
    int rst = 0;
    uint32_t rph = 0;
    int red_par = 0;
    uint32_t bcnt = 0;  // updates with gathered B couplings so far (buffer bcnt % kBD, phase (bcnt / kBD) & 1)

    for (;;) {
        __syncthreads();
        if (tid == 0) {
            int g = -1, ci = 0;
            if (!*abort_flag) {
                const unsigned t = atomicAdd(&prm.ctl->ticket, 1u);
                if (t < total_units) {
                    g = (int)(t % (unsigned)prm.n_groups);
                    ci = (int)(t / (unsigned)prm.n_groups);
                    // wait until the previous run of this group is written back
                    const unsigned long long t0 = global_ns();
                    while (true) {
                        int v;
                        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(prm.progress + g) : "memory");
                        if (v >= ci) break;
                        if (global_ns() - t0 > kWaitNs) { record_error(prm.ctl, kErrTimeout, 1); *abort_flag = 1; g = -1; break; }
                        __nanosleep(256);
                    }
                }
            }
            s_unit[0] = g; s_unit[1] = ci;
        }
        __syncthreads();
        const int g = s_unit[0], ci = s_unit[1];
        if (g < 0) break;
        const GroupDev gr = prm.groups[g];
        const SampleDev sd = prm.samples[gr.sample];
        const int N = sd.N;
        const int sw0 = ci * spu, sw1 = min(n_sweeps, sw0 + spu);
        constexpr bool useSlot = kCopyDraws<G>;  // the copy warp fills a slot for every update

        // ---- unit set-up: tables, chain metadata, amplitudes (consumers); producer starts streaming
        if (!producer) {
            for (int i = tid; i <= sd.ST; i += NCT) s_bo[i] = prm.bo[sd.tab_off + i];
            for (int i = tid; i < sd.ST; i += NCT) s_xtlo[i] = prm.xtlo[sd.tab_off + i];
            if (tid < G) {
                const int slot = gr.chain0 + tid;
                if (tid < gr.count) {
                    const int t = prm.label[slot];
                    const int r = (slot - sd.chain0) / prm.nT;
                    cE[tid] = __ldcg(prm.E + slot);
                    cBeta[tid] = (real)prm.beta[t];
                    cId[tid] = (uint32_t)((gr.sample * prm.R + r) * prm.nT + t);
                } else {
                    cE[tid] = 0.0; cBeta[tid] = real(0); cId[tid] = 0u;
                }
                cAcc[tid] = 0u; cAtt[tid] = 0ull;
            }
            const int rows = N + 2 * APAD;
            for (int i = tid; i < rows * G; i += NCT) {
                const int x = i / G - APAD, cc = i % G;
                V v; v.x = v.y = real(0);
                if (x >= 0 && x < N && cc < gr.count) {
                    const V *src = A + sd.a_off + (int64_t)(gr.chain0 - sd.chain0 + cc) * N + x;
                    const double2 t = __ldcg(reinterpret_cast<const double2 *>(src));
                    v.x = (real)t.x; v.y = (real)t.y;
                }
                as[(x + APAD) * RS + cc] = v;
            }
            named_bar(1, NCT);
        }

        if (producer) {
            // ---------------- producer warp: stream J runs of (j,k) for every update of the unit
            const int *bo_g = prm.bo + sd.tab_off;
            // identity of chain `lane` of the group (the Philox stream of its proposals): (sample, replica,
            // temperature index its slot holds)
            uint32_t pid = 0u;
            if (lane < gr.count) {
                const int slot = gr.chain0 + lane;
                pid = (uint32_t)((gr.sample * prm.R + (slot - sd.chain0) / prm.nT) * prm.nT + prm.label[slot]);
            }
            bool stop = false;
            for (int sw = sw0; sw < sw1 && !stop; ++sw) {
                const uint32_t sweep = (uint32_t)(sweep_base + sw);
                for (int u = 0; u < N / 2 && !stop; ++u) {
                    stop = __shfl_sync(0xffffffffu, *abort_flag, 0) != 0;  // warp-uniform
                    if (stop) break;
                    int j, k;
                    pair_jk(prm.seed, (uint32_t)gr.sample, sweep, (uint32_t)u, N, j, k);
                    const Ranges Rg = update_ranges(sd, bo_g, prm.mode_blk + sd.mode_off, j, k);
                    if (useSlot) {
                        // the update's slot (kBD in a ring, up to kBD updates ahead of the field warps): the random
                        // part of every chain's proposal (8 chains per block; lane = chain) and, for large N, the B_jk couplings
                        // J_j[s][{k, s-k}], s in [max(j,k), min(j,k) + N), gathered from L2 by the 32 lanes
                        const int slot = (int)(bcnt % kBD);
                        const uint32_t bph = (bcnt / kBD) & 1u;
                        ++bcnt;
                        if (mbar_wait_bounded(&bempty[slot], bph ^ 1u, prm.ctl, 4, abort_flag)) {
                            if (kCopyDraws<G> && lane < gr.count)
                                pdraw[slot * G + lane] = draw_proposal<real>(prm.seed, pid, sweep, (uint32_t)u);
                        }
                        mbar_arrive(&bfull[slot]);
                    }
                    for (int cb = Rg.ulo; cb < Rg.uhi; cb += CB, ++q, rph ^= (++rst == NST) ? 1u : 0u, rst = (rst == NST) ? 0 : rst) {
                        const int stage = rst;
                        const uint32_t ph = rph;
                        if (lane == 0) {
                            const bool ok = mbar_wait_bounded(&empty[stage], ph ^ 1u, prm.ctl, 2, abort_flag);
                            const int ce = min(cb + CB, Rg.uhi);
                            const int a0 = max(cb, Rg.jlo), a1 = min(ce, Rg.jhi);
                            const int b0 = max(cb, Rg.klo), b1 = min(ce, Rg.khi);
                            const uint32_t bj = a1 > a0 ? (uint32_t)(a1 - a0) * JS * sizeof(real) : 0u;
                            const uint32_t bk = b1 > b0 ? (uint32_t)(b1 - b0) * JS * sizeof(real) : 0u;
                            real *st_j = ring + (size_t)stage * 2 * CB * JS;
                            real *st_k = st_j + (size_t)CB * JS;
                            if (ok) mbar_arrive_expect_tx(&full[stage], bj + bk);
                            if (ok && bj) bulk_g2s(st_j + (size_t)(a0 - cb) * JS, J + (Rg.jg + (a0 - Rg.jlo)) * JS, bj, &full[stage]);
                            if (ok && bk) bulk_g2s(st_k + (size_t)(b0 - cb) * JS, J + (Rg.kg + (b0 - Rg.klo)) * JS, bk, &full[stage]);
                        }
                        __syncwarp();
                    }
                }
            }
        } else {
            // ---------------- consumer warps
            const int *mode_blk = prm.mode_blk + sd.mode_off;
            const uint32_t *binfo = prm.blkinfo + sd.blk_off;
            // update trace: absolute sweep + 1 and update to record (0 = none)
            const long long tr_at = prm.trace ? prm.ctl->trace_at : 0ll;
            const int tr_u = prm.trace ? prm.ctl->trace_update : -1;
            const real cc = (real)prm.cc;
            for (int sw = sw0; sw < sw1; ++sw) {
                const uint32_t sweep = (uint32_t)(sweep_base + sw);
                // the sweep's pair sequence, drawn once per block (every warp has read the previous sweep's
                // last entry before that update's barrier, which every thread here has passed)
                for (int i = tid; i < N / 2; i += NCT) {
                    int pj, pk;
                    pair_jk(prm.seed, (uint32_t)gr.sample, sweep, (uint32_t)i, N, pj, pk);
                    s_pair[i] = pj | (pk << 16);
                }
                named_bar(1, NCT);
                for (int u = 0; u < N / 2; ++u) {
                    const int jk = s_pair[u];
                    const int j = jk & 0xffff, k = jk >> 16;
                    const Ranges Rg = update_ranges(sd, s_bo, mode_blk, j, k);
                    // the update's slot from the copy warp (proposal draws with 8 chains per block, B couplings for
                    // large N); warp 0 puts chain c's proposal into the double-buffered table: finished from the
                    // copy warp's draw, or drawn whole
                    int pslot = 0;
                    uint32_t pph = 0u;
                    if (useSlot) {
                        pslot = (int)(bcnt % kBD);
                        pph = (bcnt / kBD) & 1u;
                        ++bcnt;
                    }
                    Proposal<real> *Pp = prop + red_par * G;
                    if (warp == 0) {
                        if constexpr (kCopyDraws<G>) {
                            const bool dok = mbar_wait_bounded(&bfull[pslot], pph, prm.ctl, 5, abort_flag);
                            if (dok && wq == 0) {
                                const V aj = as[(j + APAD) * RS + c], ak = as[(k + APAD) * RS + c];
                                Pp[c] = finish_proposal<real>(pdraw[pslot * G + c], aj, ak);
                            }
                        } else if (wq == 0) {
                            const V aj = as[(j + APAD) * RS + c], ak = as[(k + APAD) * RS + c];
                            Pp[c] = finish_proposal<real>(draw_proposal<real>(prm.seed, cId[c], sweep, (uint32_t)u), aj, ak);
                        }
                    }
                    Partials<real> pr;
                    pr.zero();
                    for (int cb = Rg.ulo; cb < Rg.uhi; cb += CB, ++q, rph ^= (++rst == NST) ? 1u : 0u, rst = (rst == NST) ? 0 : rst) {
                        const int stage = rst;
                        const uint32_t ph = rph;
                        // a chunk whose copies have landed is processed (its data are valid even after another
                        // wait gave up); a wait that gives up, or sees the abort flag, skips it
                        const bool landed = mbar_wait_bounded(&full[stage], ph, prm.ctl, 3, abort_flag);
                        const int b = cb + worker;
                        if (b < Rg.uhi && landed) {
                            const uint32_t info = __ldg(binfo + b);
                            const int st = (int)(info >> 16), xt = (int)(info & 0xffffu);
                            const int mode = ((b >= Rg.jlo && b < Rg.jhi) ? 1 : 0) | ((b >= Rg.klo && b < Rg.khi) ? 2 : 0);
                            const real *st_j = ring + (size_t)stage * 2 * CB * JS + (size_t)worker * JS;
                            const real *st_k = st_j + (size_t)CB * JS;
                            process_block_dispatch<real, RS, true>(mode, as, c, st * TS, xt * TX, j, k, N, st_j, st_k, pr);
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&empty[stage]);
                    }
                    // every warp is done with the slot (warp 0 copied the proposals out at the update's start)
                    if (useSlot) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bempty[pslot]);
                    }
                    // reduce over the workers of this warp, then across warps through shared memory
                    real v[8] = {pr.hj.x, pr.hj.y, pr.hk.x, pr.hk.y, pr.B.x, pr.B.y, pr.A.x, pr.A.y};
#pragma unroll
                    for (int o = G; o < 32; o <<= 1)
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
                    real *rb = red + (size_t)red_par * NCW * G * 8;
                    if constexpr (kSpread) {
                        // layout [warp][chain][value]: the 8 values of one (warp, chain) are consecutive, so that the
                        // reads after the barrier (32 lanes = 4 chains x 8 values of one warp) are 32 consecutive words
                        if (wq == 0) {
                                double2 *d = reinterpret_cast<double2 *>(rb + ((size_t)warp * G + c) * 8);
                                d[0] = make_double2(v[0], v[1]); d[1] = make_double2(v[2], v[3]);
                                d[2] = make_double2(v[4], v[5]); d[3] = make_double2(v[6], v[7]);
                        }
                    } else {
                        // layout [e][warp][chain]: the 8 chains of one (e, warp) are consecutive words, so both the
                        // stores below and the reads after the barrier (32 lanes = 4 warps x 8 chains) are free of
                        // bank conflicts
                        if (wq == 0) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) rb[(e * NCW + warp) * G + c] = v[e];
                        }
                    }
                    named_bar(1, NCT);
                    // Decision:
                    // - 16 chains per block: 8 lanes per chain, 4 chains per warp, warps in turn.  Lane e of a
                    //   chain's group adds value e over the warps in warp order; the group's first lane gathers
                    //   the 8 totals, decides and writes; a second barrier orders the writes before the next update;
                    // - 8 chains per block: every warp forms the same totals in the same order, takes the same
                    //   decision and writes the same values, with no second barrier.
                    if constexpr (kSpread) {
                        for (int c4 = warp * 4; c4 < G; c4 += NCW * 4) {  // warp-uniform trip count
                            const int cd = c4 + (lane >> 3), e = lane & 7;
                            const bool mine = cd < G, lead = mine && e == 0;
                            real s = 0;
                            if (mine) {
#pragma unroll
                                for (int w = 0; w < NCW; ++w) s += rb[((size_t)w * G + cd) * 8 + e];
                            }
                            real t[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) t[i] = __shfl_sync(0xffffffffu, s, (lane & ~7) | i);
                            if (lead) {
                                Partials<real> f;
                                f.hj.x = t[0]; f.hj.y = t[1]; f.hk.x = t[2]; f.hk.y = t[3];
                                f.B.x = t[4]; f.B.y = t[5]; f.A.x = t[6]; f.A.y = t[7];
                                const Proposal<real> P = Pp[cd];
                                const real dH = delta_h<real>(P, f, cc);
                                const bool live = cd < gr.count;
                                const bool acc = live && metropolis_accept(dH, cBeta[cd], P.U);
                                if (tr_at == sweep_base + sw + 1 && u == tr_u && live)
                                    trace_write<real, RS>(prm.trace, prm.n_chains, sd.a_off, sd.chain0, N, cId[cd], j, k, f, P,
                                                          dH, acc, cBeta[cd], cE[cd], as, cd);
                                if (acc) {
                                    as[(j + APAD) * RS + cd] = P.nj;
                                    as[(k + APAD) * RS + cd] = P.nk;
                                }
                                if (live) {
                                    if (acc) { cE[cd] += (double)dH; cAcc[cd] += 1u; }
                                    cAtt[cd] += 1ull;
                                }
                            }
                        }
                    } else {
                        // lane (c, wq) adds the partials of warps wq, wq + WPW, ...: the trip count is the
                        // same on every lane (predicated body), so the warp is converged at the shuffles
                        real t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
                        for (int w0 = 0; w0 < NCW; w0 += WPW) {
                            const int w = w0 + wq;
                            if (w < NCW) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) t[e] += rb[(e * NCW + w) * G + c];
                            }
                        }
                        __syncwarp();
#pragma unroll
                        for (int o = G; o < 32; o <<= 1)
#pragma unroll
                            for (int e = 0; e < 8; ++e) t[e] += __shfl_xor_sync(0xffffffffu, t[e], o);
                        if (wq == 0) {
                            Partials<real> f;
                            f.hj.x = t[0]; f.hj.y = t[1]; f.hk.x = t[2]; f.hk.y = t[3];
                            f.B.x = t[4]; f.B.y = t[5]; f.A.x = t[6]; f.A.y = t[7];
                            const Proposal<real> P = Pp[c];
                            const real dH = delta_h<real>(P, f, cc);
                            const bool acc = (c < gr.count) && metropolis_accept(dH, cBeta[c], P.U);
                            if (tr_at == sweep_base + sw + 1 && u == tr_u && warp == 0 && c < gr.count)
                                trace_write<real, RS>(prm.trace, prm.n_chains, sd.a_off, sd.chain0, N, cId[c], j, k, f, P, dH, acc,
                                                      cBeta[c], cE[c], as, c);
                            if (acc) {
                                as[(j + APAD) * RS + c] = P.nj;
                                as[(k + APAD) * RS + c] = P.nk;
                            }
                            if (warp == 0 && c < gr.count) {
                                if (acc) { cE[c] += (double)dH; cAcc[c] += 1u; }
                                cAtt[c] += 1ull;
                            }
                        }
                    }
                    red_par ^= 1;
                    if constexpr (kSpread) named_bar(1, NCT);
                    else __syncwarp();
                }
                // interior measurement point: snapshot amplitudes and energies
                const long long done = sweep_base + sw + 1;
                if (prm.measure_every > 0 && done % prm.measure_every == 0 && sw + 1 < n_sweeps) {
                    named_bar(1, NCT);
                    // snapshot index = number of measurement points in (sweep_base, done], minus one
                    const int kk = (int)(done / prm.measure_every - sweep_base / prm.measure_every - 1);
                    if (kk >= 0 && kk < prm.n_snap_max) {
                        V *dst = reinterpret_cast<V *>(prm.snap_a) + (int64_t)kk * prm.a_total + sd.a_off +
                                 (int64_t)(gr.chain0 - sd.chain0) * N;
                        for (int i = tid; i < N * gr.count; i += NCT) {
                            const int cc2 = i / N, x = i % N;
                            dst[(int64_t)cc2 * N + x] = as[(x + APAD) * RS + cc2];
                        }
                        if (tid < gr.count) prm.snap_E[(int64_t)kk * prm.n_chains + gr.chain0 + tid] = cE[tid];
                    }
                    named_bar(1, NCT);
                }
            }
            // ---- write back the group's state and counters
            named_bar(1, NCT);
            for (int i = tid; i < N * gr.count; i += NCT) {
                const int cc2 = i / N, x = i % N;
                V *dst = A + sd.a_off + (int64_t)(gr.chain0 - sd.chain0 + cc2) * N + x;
                __stcg(dst, as[(x + APAD) * RS + cc2]);
            }
            if (tid < gr.count) {
                const int slot = gr.chain0 + tid;
                __stcg(prm.E + slot, cE[tid]);
                prm.mc_acc[slot] += cAcc[tid];
                prm.mc_att[slot] += cAtt[tid];
            }
            __threadfence();
            named_bar(1, NCT);
            if (tid == 0) {
                asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(prm.progress + g), "r"(ci + 1) : "memory");
            }
        }
    }
    // never leave bulk copies in flight behind an exiting block (only possible after an abort)
    if (producer && lane == 0) {
        const uint32_t first = q > (uint32_t)NST ? q - NST : 0u;
        for (uint32_t qq = first; qq < q; ++qq) {
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(&full[qq % NST], (qq / NST) & 1u) && global_ns() - t0 < kWaitNs) {
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Field-only kernel: the same block arithmetic with J read straight from global memory; one thread
// block per group of the chosen sample.  Output: 8 doubles per chain (h_j, h_k, B_jk, A_jk).
template <typename real, int G>
__global__ void fields_kernel(FieldsParams prm) {
    using V = typename vec2<real>::type;
    constexpr int RS = RowStride<real, G>::value, NCW = 4, WPW = 32 / G, NW = NCW * WPW;
    extern __shared__ __align__(128) unsigned char smem[];
    V *as = reinterpret_cast<V *>(smem);
    const GroupDev gr = prm.groups[prm.group0 + blockIdx.x];
    const SampleDev sd = prm.samples[gr.sample];
    const int N = sd.N, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int c = lane % G, worker = warp * WPW + lane / G;
    const V *A = reinterpret_cast<const V *>(prm.a);
    real *red = reinterpret_cast<real *>(smem + (size_t)(N + 2 * APAD) * RS * sizeof(V));
    for (int i = tid; i < (N + 2 * APAD) * G; i += blockDim.x) {
        const int x = i / G - APAD, cc = i % G;
        V v; v.x = v.y = real(0);
        if (x >= 0 && x < N && cc < gr.count) v = A[sd.a_off + (int64_t)(gr.chain0 - sd.chain0 + cc) * N + x];
        as[(x + APAD) * RS + cc] = v;
    }
    __syncthreads();
    const int j = prm.j, k = prm.k;
    const Ranges Rg = update_ranges(sd, prm.bo + sd.tab_off, prm.mode_blk + sd.mode_off, j, k);
    const real *J = reinterpret_cast<const real *>(prm.J);
    Partials<real> pr;
    pr.zero();
    for (int b = Rg.ulo + worker; b < Rg.uhi; b += NW) {
        const uint32_t info = prm.blkinfo[sd.blk_off + b];
        const int st = (int)(info >> 16), xt = (int)(info & 0xffffu);
        const int mode = ((b >= Rg.jlo && b < Rg.jhi) ? 1 : 0) | ((b >= Rg.klo && b < Rg.khi) ? 2 : 0);
        const real *Jj = J + (Rg.jg + (b - Rg.jlo)) * JStride<real>::value;
        const real *Jk = J + (Rg.kg + (b - Rg.klo)) * JStride<real>::value;
        process_block_dispatch<real, RS, true>(mode, as, c, st * TS, xt * TX, j, k, N, Jj, Jk, pr);
    }
    real v[8] = {pr.hj.x, pr.hj.y, pr.hk.x, pr.hk.y, pr.B.x, pr.B.y, pr.A.x, pr.A.y};
#pragma unroll
    for (int o = G; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
    if (lane < G)
        for (int e = 0; e < 8; ++e) red[(warp * G + c) * 8 + e] = v[e];
    __syncthreads();
    if (tid < G * 8 && tid / 8 < gr.count) {
        const int cc = tid / 8, e = tid % 8;
        double t = 0.0;
        for (int w = 0; w < NCW; ++w) t += (double)red[(w * G + cc) * 8 + e];
        prm.out[(int64_t)(gr.chain0 - sd.chain0 + cc) * 8 + e] = t;
    }
}

// ------------------------------------------------------------------------------------------------
// Full energy (resync).  With the partial fields h^>_x = sum_{m > x} conj(a_m) acc^>_x[x+m], where acc^>
// keeps only the pairs {p, q} of row x+m whose smaller mode (the block column) exceeds x,
//     H = -cc sum_x Re( conj(a_x) h^>_x ),
// which visits every quadruplet once, at its smallest mode x (partner m: the largest; the pair {p, q} of
// the two middle modes has p > x).  A group's share is split over prm.parts thread blocks, each writing per-chain FP64
// sums to prm.part, and energy_sum_kernel adds the parts in order.  With renorm != 0, renorm_kernel first rescales every
// chain onto sum |a|^4 = N.  FP32 chains: energy_tile_kernel (pt_energy.cu), but for many groups of small N (energy_tiles).
// Those and FP64: energy_kernel, whose work items are (mode, block); it waits on coupling loads from L2, so it runs about 8
// blocks per SM in all.
template <typename real, int G>
__global__ void __launch_bounds__(256) renorm_kernel(EnergyParams prm) {
    using V = typename vec2<real>::type;
    const GroupDev gr = prm.groups[blockIdx.x];
    const SampleDev sd = prm.samples[gr.sample];
    const int N = sd.N, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    V *Ag = reinterpret_cast<V *>(prm.a);
    // sum |a|^4 per chain in FP64 (one warp per chain, round robin), then the rescaled amplitudes
    for (int cc = warp; cc < gr.count; cc += 8) {
        V *a = Ag + sd.a_off + (int64_t)(gr.chain0 - sd.chain0 + cc) * N;
        double s4 = 0.0;
        for (int x = lane; x < N; x += 32) {
            const V v = a[x];
            const double u = (double)v.x * v.x + (double)v.y * v.y;
            s4 += u * u;
        }
        for (int o = 16; o; o >>= 1) s4 += __shfl_xor_sync(0xffffffffu, s4, o);
        if (lane == 0 && (!(s4 > 0.0) || !isfinite(s4))) record_error(prm.ctl, kErrNaN, 10);
        const double f = sqrt(sqrt((double)N / s4));
        for (int x = lane; x < N; x += 32) {
            V v = a[x];
            v.x = (real)((double)v.x * f); v.y = (real)((double)v.y * f);
            a[x] = v;
        }
    }
}

template <typename real, int G>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 3 : 2) energy_kernel(EnergyParams prm) {
    using V = typename vec2<real>::type;
    constexpr int RS = RowStride<real, G>::value, NCW = 8, WPW = 32 / G, NW = NCW * WPW;
    extern __shared__ __align__(128) unsigned char smem[];
    const int part = (int)(blockIdx.x % (unsigned)prm.parts);
    const GroupDev gr = prm.groups[blockIdx.x / (unsigned)prm.parts];
    const SampleDev sd = prm.samples[gr.sample];
    const int N = sd.N, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int c = lane % G, worker = warp * WPW + lane / G;
    V *as = reinterpret_cast<V *>(smem);
    double *dred = reinterpret_cast<double *>(smem + (size_t)(N + 2 * APAD) * RS * sizeof(V));
    V *Ag = reinterpret_cast<V *>(prm.a);
    for (int i = tid; i < (N + 2 * APAD) * G; i += blockDim.x) {
        const int x = i / G - APAD, cc = i % G;
        V v; v.x = v.y = real(0);
        if (x >= 0 && x < N && cc < gr.count) v = Ag[sd.a_off + (int64_t)(gr.chain0 - sd.chain0 + cc) * N + x];
        as[(x + APAD) * RS + cc] = v;
    }
    __syncthreads();
    const real *J = reinterpret_cast<const real *>(prm.J);
    const int *bo = prm.bo + sd.tab_off;
    const int *mode_blk = prm.mode_blk + sd.mode_off;
    const int *ebo = prm.ebo + sd.mode_off;  // prefix over x of the blocks with rows s > 2x
    const int total = ebo[N];
    double e = 0.0;
    int x = 0;
    for (int it = part * NW + worker; it < total; it += NW * prm.parts) {
        while (ebo[x + 1] <= it) ++x;
        const int stlo = x / TS;
        const int sta = (2 * x + 1) / TS;
        const int b = bo[sta] + (it - ebo[x]);
        const uint32_t info = prm.blkinfo[sd.blk_off + b];
        const int st = (int)(info >> 16), xt = (int)(info & 0xffffu);
        const real *Jx = J + (sd.J_off + mode_blk[x] + (b - bo[stlo])) * JStride<real>::value;
        const int s0 = st * TS, x0 = xt * TX;
        if (x0 + TX - 1 <= x) continue;  // every pair of the block has its smaller mode <= x
        V ax[TX], ay[TS + TX - 1], acc[TS];
#pragma unroll
        for (int i = 0; i < TX; ++i) ax[i] = as[(x0 + i + APAD) * RS + c];
        const int ybase = s0 - x0 - (TX - 1) + APAD;
#pragma unroll
        for (int d = 0; d < TS + TX - 1; ++d) ay[d] = as[(ybase + d) * RS + c];
#pragma unroll
        for (int r = 0; r < TS; ++r) acc[r].x = acc[r].y = real(0);
#pragma unroll
        for (int i = 0; i < TX; ++i) {
            if (x0 + i <= x) continue;  // pairs whose smaller mode is <= x: counted at that mode
            JRow<real> jc;
            jc.load(Jx + i * TS);
#pragma unroll
            for (int r = 0; r < TS; ++r) caxpy(acc[r], jc.v[r], cmul(ax[i], ay[r - i + TX - 1]));
        }
        const V axx = as[(x + APAD) * RS + c];
        real blk = real(0);
#pragma unroll
        for (int r = 0; r < TS; ++r) {
            const int m = s0 + r - x;
            if (m > x && m < N) {
                const V zz = cmul(axx, as[(m + APAD) * RS + c]);  // z_{x,m}
                blk += zz.x * acc[r].x + zz.y * acc[r].y;          // Re(conj(z) acc)
            }
        }
        e += (double)blk;
    }
    for (int o = G; o < 32; o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane < G) dred[warp * G + c] = e;
    __syncthreads();
    if (tid < gr.count) {
        double t = 0.0;
        for (int w = 0; w < NCW; ++w) t += dred[w * G + tid];
        prm.part[((size_t)(blockIdx.x / (unsigned)prm.parts) * prm.parts + part) * 32 + tid] = t;
    }
}

// E = -cc (sum of the parts, in part order) per chain of a group; one thread per chain.
__global__ void energy_sum_kernel(EnergyParams prm) {
    const GroupDev gr = prm.groups[blockIdx.x];
    const int c = threadIdx.x;
    if (c >= gr.count) return;
    double t = 0.0;
    for (int p = 0; p < prm.parts; ++p) t += prm.part[((size_t)blockIdx.x * prm.parts + p) * 32 + c];
    const double E = -prm.cc * t;
    if (!isfinite(E)) record_error(prm.ctl, kErrNaN, 11);
    if (prm.E_out) prm.E_out[gr.chain0 + c] = E;
    if (prm.E_state) prm.E_state[gr.chain0 + c] = E;
}

// ------------------------------------------------------------------------------------------------
// host launchers
// Opt-in shared memory per block of the current device.
static size_t smem_limit() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return (size_t)v;
}

template <typename real, int G, int NCW>
static cudaError_t launch_sweep_t(const SweepParams &p, int grid, cudaStream_t s) {
    SweepParams q = p;
    q.nst = sweep_stages<real, G, NCW>(p.maxN, smem_limit());
    if (q.nst < kNstMin) return cudaErrorInvalidConfiguration;
    const size_t sm = sweep_smem_bytes<real, G, NCW>(p.maxN, q.nst);
    cudaError_t e = cudaFuncSetAttribute(sweep_kernel<real, G, NCW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    sweep_kernel<real, G, NCW><<<grid, (NCW + 1) * 32, sm, s>>>(q);
    return cudaGetLastError();
}

template <typename real, int G, int NCW>
static int occupancy_t(int maxN) {
    const int nst = sweep_stages<real, G, NCW>(maxN, smem_limit());
    if (nst < kNstMin) return 0;
    const size_t sm = sweep_smem_bytes<real, G, NCW>(maxN, nst);
    if (cudaFuncSetAttribute(sweep_kernel<real, G, NCW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sweep_kernel<real, G, NCW>, (NCW + 1) * 32, sm) != cudaSuccess)
        return 0;
    return nb;
}

#define PT_SWEEP_VARIANTS(X)                                          \
    X(double, 8, 7) X(double, 16, 3)

bool sweep_variant_exists(bool dbl, int G, int ncw) {
#define X(T, g, n) if (dbl == (sizeof(T) == 8) && G == g && ncw == n) return true;
    PT_SWEEP_VARIANTS(X)
#undef X
    return false;
}

cudaError_t launch_sweep(bool dbl, int G, int ncw, const SweepParams &p, int grid, cudaStream_t s) {
#define X(T, g, n) \
    if (dbl == (sizeof(T) == 8) && G == g && ncw == n) return launch_sweep_t<T, g, n>(p, grid, s);
    PT_SWEEP_VARIANTS(X)
#undef X
    return cudaErrorInvalidValue;
}

int sweep_occupancy(bool dbl, int G, int ncw, int maxN) {
#define X(T, g, n) \
    if (dbl == (sizeof(T) == 8) && G == g && ncw == n) return occupancy_t<T, g, n>(maxN);
    PT_SWEEP_VARIANTS(X)
#undef X
    return 0;
}

template <typename real, int G>
static cudaError_t launch_fields_t(const FieldsParams &p, int ngroups, int maxN, cudaStream_t s) {
    using V = typename vec2<real>::type;
    const size_t sm = (size_t)(maxN + 2 * APAD) * RowStride<real, G>::value * sizeof(V) + 4 * G * 8 * sizeof(real) + 64;
    cudaError_t e = cudaFuncSetAttribute(fields_kernel<real, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    fields_kernel<real, G><<<ngroups, 128, sm, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_fields(bool dbl, int G, const FieldsParams &p, int ngroups, int maxN, cudaStream_t s) {
    if (!dbl) {
        if (G == 8) return launch_fields_t<float, 8>(p, ngroups, maxN, s);
        if (G == 16) return launch_fields_t<float, 16>(p, ngroups, maxN, s);
        if (G == 32) return launch_fields_t<float, 32>(p, ngroups, maxN, s);
    } else {
        if (G == 8) return launch_fields_t<double, 8>(p, ngroups, maxN, s);
        if (G == 16) return launch_fields_t<double, 16>(p, ngroups, maxN, s);
    }
    return cudaErrorInvalidValue;
}

template <typename real, int G>
static cudaError_t launch_energy_t(const EnergyParams &p, int ngroups, int maxN, cudaStream_t s) {
    using V = typename vec2<real>::type;
    const size_t sm = (size_t)(maxN + 2 * APAD) * RowStride<real, G>::value * sizeof(V) + 8 * G * sizeof(double) + 64;
    cudaError_t e = p.tiles ? cudaSuccess : cudaFuncSetAttribute(energy_kernel<real, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    if (p.parts < 1 || p.parts > kEnergyPartsMax || !p.part) return cudaErrorInvalidValue;
    if (p.renorm) {
        renorm_kernel<real, G><<<ngroups, 256, 0, s>>>(p);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (p.tiles) e = launch_energy_tiles(G, p, ngroups, s);
    else {
        energy_kernel<real, G><<<ngroups * p.parts, 256, sm, s>>>(p);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    energy_sum_kernel<<<ngroups, 32, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_energy(bool dbl, int G, const EnergyParams &p, int ngroups, int maxN, cudaStream_t s) {
    if (!dbl) {
        if (G == 8) return launch_energy_t<float, 8>(p, ngroups, maxN, s);
        if (G == 16) return launch_energy_t<float, 16>(p, ngroups, maxN, s);
        if (G == 32) return launch_energy_t<float, 32>(p, ngroups, maxN, s);
    } else {
        if (G == 8) return launch_energy_t<double, 8>(p, ngroups, maxN, s);
        if (G == 16) return launch_energy_t<double, 16>(p, ngroups, maxN, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace ptgb
