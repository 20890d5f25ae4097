// pt_comb.cu -- the J-sharing FP32 Metropolis sweep of the comb graph (sm_103a; arXiv 2511.13508, Sec. III.A).
//
// Local field of the updated modes.  With z_P = a_x a_y for the pair P = {x, y}, the field of mode l factorises over
// the pair sum s = x + y:
//     h_l = sum_s conj(a_{s-l}) acc_l[s],     acc_l[s] = sum_{P : x+y=s} J_l[s][P] z_P,
// so one product z_P feeds both fields of a pair update (j,k), and all chains of a disorder sample read the same
// couplings: the J rows stream L2 -> shared memory by bulk copies, while the amplitudes of the group's G chains stay
// resident.  A group runs on one thread block, or, when there are fewer groups than SMs, on a cluster of C blocks:
// each block streams and evaluates every C-th chunk of an update and sends its share of the energy change to the others.
//
// What bounds it: FP32 issue.  With three warps per scheduler the kernel issues about one instruction in two cycles
// whatever the mix, half of them paired FP32 multiply-adds, so instructions outside the blocks are what can be saved:
// a lane folds its field sums with the proposal into its share of dH (one value to reduce, not eight), and one barrier
// per update orders the shares before every warp's own copy of the decision.
// Measured on GB300, us per sweep, against eight sums reduced per chain behind two barriers and one block per group with
// whole sweeps as work units: N = 256, 16 samples of 96 chains, 8 sweeps a launch 2300 -> 2127 (the finer units); one such
// sample 1680 -> 428 (clusters of 8); N = 64, 64 samples of 64 chains 163 -> 161; ragged N = 32 ... 128, 96 samples of 48
// chains 510 -> 494 in launches of 64 sweeps (505 of 8, 516 of one).
#include <cstdint>
#include "pt_bulk.cuh"
#include "pt_common.cuh"
#include "pt_kernels.h"
#include "pt_move.cuh"

namespace ptgb {

namespace {

constexpr int kJS = JStride<float>::value;  // floats per stored block

// Row stride of the amplitude table [x + APAD][chain]: one pad chain at 8 chains, so that four workers reading rows 8
// apart meet distinct bank halves.
template <int G> __host__ __device__ constexpr int row_stride() { return G == 8 ? G + 1 : G; }

__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 4 bytes into a peer block's shared memory, counted on the mbarrier at the same place there
__device__ __forceinline__ void send_async(uint32_t at, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at), "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}

// ------------------------------------------------------------------------------------------------
// Packed-FP32 block arithmetic.  Rows are taken in pairs (r, r+1) and every quantity is a float2 over the two rows, so
// each instruction does two fused multiply-adds: with
//     sx = (Re a_x, Re a_x), sy = (Im a_x, Im a_x)                  (splats of a_x in registers)
//     WX = (Re a_y, Re a_{y+1}), WY = (Im a_y, Im a_{y+1})          (window table awin, y = s - x)
// the pair products of rows (s, s+1) at column x are
//     Re z = sx WX - sy WY,   Im z = sx WY + sy WX,
// and a field row pair accumulates acc += (J[s][x], J[s+1][x]) z with the column-major J block supplying
// the coupling pair directly.  Two FMUL2 + two FFMA2 make 2 products; one FFMA2 per field per component
// accumulates them: 2 instructions per coupling term when both fields use the block, 3 otherwise.
struct PartialsX2 {
    float2 hjx, hjy, hjyn, hkx, hky, hkyn;  // h = (hx.0 + hx.1, (hy.0 + hy.1) - (hyn.0 + hyn.1))
    float2 B, A;
    __device__ __forceinline__ void zero() {
        hjx = hjy = hjyn = hkx = hky = hkyn = B = A = make_float2(0.f, 0.f);
    }
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

template <int G, int MODE>
__device__ __forceinline__ void process_block_x2(const float2 *__restrict__ as, const float4 *__restrict__ awin,
                                                 int c, int s0, int x0, int j, int k, const float *Jj,
                                                 const float *Jk, PartialsX2 &p) {
    constexpr int RS = row_stride<G>();
    // Column i = 2h + pi pairs rows (2q, 2q+1) with the window starting at y-offset d = 2q - i + 7, of parity
    // 1 - pi: the columns run in two passes by parity, each holding the 7 windows of its parity
    // (d = 2m + 1 - pi, m = q - h + 3), so that only 7 windows are live at a time.
    const int ybase = s0 - x0 - (TX - 1) + APAD;
    float2 ajx[TS / 2], ajy[TS / 2], akx[TS / 2], aky[TS / 2];
#pragma unroll
    for (int q = 0; q < TS / 2; ++q) ajx[q] = ajy[q] = akx[q] = aky[q] = f2(0.f, 0.f);
#pragma unroll
    for (int pi = 0; pi < 2; ++pi) {
        float2 wx[7], wy[7];
#pragma unroll
        for (int m = 0; m < 7; ++m) {
            const float4 w = awin[(ybase + 2 * m + 1 - pi) * G + c];
            wx[m] = f2(w.x, w.y);
            wy[m] = f2(w.z, w.w);
        }
#pragma unroll
        for (int h = 0; h < TX / 2; ++h) {
            const int i = 2 * h + pi;
            // splats of a_x in registers (register moves cost less than the shared-memory bandwidth of a table)
            const float2 axv = as[(x0 + i + APAD) * RS + c];
            const float2 sx = f2(axv.x, axv.x), sy = f2(axv.y, axv.y), nsy = f2(-axv.y, -axv.y);
            float2 jp[TS / 2], kp[TS / 2];
            if (MODE & 1) {
                const float4 a = *reinterpret_cast<const float4 *>(Jj + i * TS), b = *reinterpret_cast<const float4 *>(Jj + i * TS + 4);
                jp[0] = f2(a.x, a.y); jp[1] = f2(a.z, a.w); jp[2] = f2(b.x, b.y); jp[3] = f2(b.z, b.w);
            }
            if (MODE & 2) {
                const float4 a = *reinterpret_cast<const float4 *>(Jk + i * TS), b = *reinterpret_cast<const float4 *>(Jk + i * TS + 4);
                kp[0] = f2(a.x, a.y); kp[1] = f2(a.z, a.w); kp[2] = f2(b.x, b.y); kp[3] = f2(b.z, b.w);
            }
            float2 tx[TS / 2], ty[TS / 2], zx[TS / 2], zy[TS / 2];
#pragma unroll
            for (int q = 0; q < TS / 2; ++q) {
                const int m = q - h + 3;
                tx[q] = __fmul2_rn(nsy, wy[m]);
                ty[q] = __fmul2_rn(sy, wx[m]);
            }
#pragma unroll
            for (int q = 0; q < TS / 2; ++q) {
                const int m = q - h + 3;
                zx[q] = __ffma2_rn(sx, wx[m], tx[q]);
                zy[q] = __ffma2_rn(sx, wy[m], ty[q]);
            }
#pragma unroll
            for (int q = 0; q < TS / 2; ++q) {
                if (MODE & 1) { ajx[q] = __ffma2_rn(jp[q], zx[q], ajx[q]); ajy[q] = __ffma2_rn(jp[q], zy[q], ajy[q]); }
                if (MODE & 2) { akx[q] = __ffma2_rn(kp[q], zx[q], akx[q]); aky[q] = __ffma2_rn(kp[q], zy[q], aky[q]); }
            }
        }
    }
    // close the rows: h += conj(m) acc with m = a_{s-l} for the row pair (s, s+1) from the window table
#pragma unroll
    for (int q = 0; q < TS / 2; ++q) {
        if (MODE & 1) {
            const float4 w = awin[(s0 + 2 * q - j + APAD) * G + c];
            const float2 mx = f2(w.x, w.y), my = f2(w.z, w.w);
            p.hjx = __ffma2_rn(mx, ajx[q], p.hjx);
            p.hjx = __ffma2_rn(my, ajy[q], p.hjx);
            p.hjy = __ffma2_rn(mx, ajy[q], p.hjy);
            p.hjyn = __ffma2_rn(my, ajx[q], p.hjyn);
        }
        if (MODE & 2) {
            const float4 w = awin[(s0 + 2 * q - k + APAD) * G + c];
            const float2 mx = f2(w.x, w.y), my = f2(w.z, w.w);
            p.hkx = __ffma2_rn(mx, akx[q], p.hkx);
            p.hkx = __ffma2_rn(my, aky[q], p.hkx);
            p.hky = __ffma2_rn(mx, aky[q], p.hky);
            p.hkyn = __ffma2_rn(my, akx[q], p.hkyn);
        }
    }
    if (MODE & 1) {
        // A_jk is the accumulator of row j+k
        const int rs = j + k - s0;
        if (rs >= 0 && rs < TS) {
#pragma unroll
            for (int q = 0; q < TS / 2; ++q) {
                if (rs == 2 * q) { p.A.x += ajx[q].x; p.A.y += ajy[q].x; }
                if (rs == 2 * q + 1) { p.A.x += ajx[q].y; p.A.y += ajy[q].y; }
            }
        }
    }
}


struct Ranges {  // block ranges of an update: the runs of j and k in the sample's block list
    int jlo, jhi, klo, khi, ulo, uhi;
    int64_t jg, kg;  // first block of j's / k's run in the coupling store
};
__device__ __forceinline__ Ranges update_ranges(const SampleDev &sd, const int *bo, const int *mode_blk, int j, int k) {
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

// The coupling J_j[s][{k, s-k}] of quadruplet {j, s-j, k, s-k} (0 where the store holds no such entry): column
// min(k, s-k) of row s in mode j's run, read from global memory (in L2: the run streams for the same update).
__device__ __forceinline__ float b_coupling(const float *__restrict__ J, const int *bo, const int *xtlo, const Ranges &Rg, int s, int k) {
    const int y = s - k, x = y < k ? y : k, st = s / TS, xt = x / TX, xi = xt - xtlo[st];
    if (xi < 0 || xi >= bo[st + 1] - bo[st]) return 0.f;
    return __ldg(J + (Rg.jg + (bo[st] + xi - Rg.jlo)) * kJS + (x - xt * TX) * TS + (s - st * TS));
}

// Ring depth: as many stages as fit next to the tables of the largest N (up to kNstMax), so that a chunk's copies are
// issued several chunks ahead of its use.  Per-update slots (B_jk couplings, proposal draws): kBD updates ahead.
constexpr int kNstMax = 6, kNstMin = 2, kBD = 4;

template <int G, int NCW> struct CombShape {
    static constexpr int WPW = 32 / G;       // workers of a warp
    static constexpr int CB = NCW * WPW;     // workers of a block, blocks of a chunk
    static constexpr size_t stage_bytes = (size_t)2 * CB * kJS * sizeof(float);
};

struct CombSmem {
    size_t bars, win, amp, bval, draws, part, xpart, pair, ints, ring, total;
};
template <int G, int NCW, int C> __host__ __device__ CombSmem comb_smem(int maxN, int nst) {
    CombSmem m;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o += (bytes + 15) / 16 * 16; return at; };
    m.bars = take((2 * (kNstMax + kBD) + 2) * sizeof(uint64_t));
    m.win = take((size_t)(maxN + 2 * APAD) * G * sizeof(float4));
    m.amp = take((size_t)(maxN + 2 * APAD) * row_stride<G>() * sizeof(float2));
    m.bval = take((size_t)kBD * maxN * sizeof(float));
    m.draws = take((size_t)kBD * G * sizeof(ProposalDraw<float>));
    m.part = take((size_t)2 * NCW * G * sizeof(float));
    m.xpart = take(C > 1 ? (size_t)2 * C * G * sizeof(float) : 0);
    m.pair = take((size_t)(maxN / 2) * sizeof(int));
    m.ints = take((size_t)(2 * 129 + 4) * sizeof(int));
    m.ring = (o + 127) / 128 * 128;
    m.total = m.ring + (size_t)nst * CombShape<G, NCW>::stage_bytes;
    return m;
}

}  // namespace

// NCW field warps and a copy warp.  A lane is (chain c = lane % G, worker lane / G of its warp); worker w takes block w of
// every chunk of CB blocks.  The copy warp streams the J runs of j and k into a ring of nst stages and fills one slot
// per update with the B_jk couplings and the random part of every chain's proposal.  Work units (group, run of sweeps)
// come from a ticket counter; a unit waits (bounded) until the previous run of its group has been written back.  A run need
// not end with a sweep: the launcher cuts each group's updates into as many equal runs as balance the SMs best.
template <int G, int NCW, int C>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) comb_sweep_kernel(SweepParams p) {
    using Sh = CombShape<G, NCW>;
    constexpr int RS = row_stride<G>(), CB = Sh::CB, WPW = Sh::WPW, NCT = NCW * 32;
    const int NST = p.nst;
    extern __shared__ __align__(128) unsigned char smem[];
    const CombSmem lay = comb_smem<G, NCW, C>(p.maxN, NST);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + lay.bars);
    uint64_t *empty = full + kNstMax, *bfull = empty + kNstMax, *bempty = bfull + kBD, *pbar = bempty + kBD;
    float4 *win = reinterpret_cast<float4 *>(smem + lay.win);
    float2 *amp = reinterpret_cast<float2 *>(smem + lay.amp);
    float *bval = reinterpret_cast<float *>(smem + lay.bval);  // [kBD][maxN]: s = max(j,k) + i
    ProposalDraw<float> *draws = reinterpret_cast<ProposalDraw<float> *>(smem + lay.draws);  // [kBD][G]
    float *part = reinterpret_cast<float *>(smem + lay.part);    // [2][NCW][G]: the warps' shares of -dH/cc
    float *xpart = reinterpret_cast<float *>(smem + lay.xpart);  // [2][C][G]: the blocks' shares (clusters)
    int *s_pair = reinterpret_cast<int *>(smem + lay.pair);    // (j | k << 16) of every update of the sweep
    int *s_bo = reinterpret_cast<int *>(smem + lay.ints), *s_xtlo = s_bo + 129;
    volatile int *s_unit = s_xtlo + 129;  // group, run, abort
    volatile int *abort_flag = s_unit + 2;
    float *ring = reinterpret_cast<float *>(smem + lay.ring);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool producer = warp == NCW;
    const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;
    const int c = lane % G, wq = lane / G, worker = warp * WPW + wq;

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], NCW); }
        for (int i = 0; i < kBD; ++i) { mbar_init(&bfull[i], 32); mbar_init(&bempty[i], NCW); }
        mbar_init(&pbar[0], 1); mbar_init(&pbar[1], 1);
        s_unit[2] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    auto sync_all = [&]() {
        if (C > 1) cluster_sync_all();
        else __syncthreads();
    };

    const long long sweep_base = p.ctl->sweep_base;
    const int n_sweeps = p.n_sweeps;
    const unsigned units = (unsigned)p.runs * (unsigned)p.n_groups;
    const float *J = reinterpret_cast<const float *>(p.J);
    float2 *A = reinterpret_cast<float2 *>(p.a);
    uint32_t q = 0;  // chunks so far (ring position); stage and phase advance with it, without a division
    int rst = 0;
    uint32_t rph = 0;
    uint32_t bcnt = 0;  // updates so far: slot bcnt % kBD, phase (bcnt / kBD) & 1
    uint32_t upd = 0;   // updates so far (field warps): share buffer upd & 1, phase (upd >> 1) & 1

    for (;;) {
        sync_all();
        if (tid == 0 && rank == 0) {
            int g = -1, ci = 0;
            if (!*abort_flag) {
                const unsigned t = atomicAdd(&p.ctl->ticket, 1u);
                if (t < units) {
                    g = (int)(t % (unsigned)p.n_groups);
                    ci = (int)(t / (unsigned)p.n_groups);
                    const unsigned long long t0 = global_ns();
                    while (true) {
                        int v;
                        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p.progress + g) : "memory");
                        if (v >= ci) break;
                        if (global_ns() - t0 > kWaitNs) { record_error(p.ctl, kErrTimeout, 1); g = -1; break; }
                        __nanosleep(256);
                    }
                }
            }
            if (C == 1) { s_unit[0] = g; s_unit[1] = ci; }
            else {
                for (int r = 0; r < C; ++r)
                    asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(cluster_map(smem_u32((const void *)s_unit), r)), "r"(g), "r"(ci)
                                 : "memory");
            }
        }
        sync_all();
        const int g = s_unit[0], ci = s_unit[1];
        if (g < 0) break;
        const GroupDev gr = p.groups[g];
        const SampleDev sd = p.samples[gr.sample];
        const int N = sd.N, half = N / 2;
        // updates [n0, n1) of the group's n_sweeps * half
        const int n0 = (int)((long long)n_sweeps * half * ci / p.runs), n1 = (int)((long long)n_sweeps * half * (ci + 1) / p.runs);
        const int *mode_blk = p.mode_blk + sd.mode_off;
        // identity of chain c (the Philox stream of its proposals): (sample, replica, temperature its slot holds)
        uint32_t id = 0u;
        int temp = 0;
        if (c < gr.count) {
            const int slot = gr.chain0 + c;
            temp = p.label[slot];
            id = (uint32_t)((gr.sample * p.R + (slot - sd.chain0) / p.nT) * p.nT + temp);
        }

        if (producer) {
            const int *bo_g = p.bo + sd.tab_off, *xtlo_g = p.xtlo + sd.tab_off;
            int sw = n0 / half, u = n0 - sw * half;
            {
                for (int n = n0; n < n1; ++n, u = u + 1 == half ? (++sw, 0) : u + 1) {
                    const uint32_t sweep = (uint32_t)(sweep_base + sw);
                    if (__shfl_sync(0xffffffffu, *abort_flag, 0) != 0) break;  // warp-uniform
                    int j, k;
                    pair_jk(p.seed, (uint32_t)gr.sample, sweep, (uint32_t)u, N, j, k);
                    const Ranges Rg = update_ranges(sd, bo_g, mode_blk, j, k);
                    // the update's slot: proposal draws (lane = chain), B_jk couplings for s in [max(j,k), min(j,k) + N)
                    const int slot = (int)(bcnt % kBD);
                    const uint32_t bph = (bcnt / kBD) & 1u;
                    ++bcnt;
                    if (mbar_wait_bounded(&bempty[slot], bph ^ 1u, p.ctl, 4, abort_flag)) {
                        if (lane < gr.count) draws[slot * G + lane] = draw_proposal<float>(p.seed, id, sweep, (uint32_t)u);
                        const int s_lo = max(j, k), n = min(j, k) + N - s_lo;
                        for (int i = lane; i < n; i += 32) bval[slot * p.maxN + i] = b_coupling(J, bo_g, xtlo_g, Rg, s_lo + i, k);
                    }
                    mbar_arrive(&bfull[slot]);
                    for (int cb = Rg.ulo + rank * CB; cb < Rg.uhi; cb += C * CB, ++q, rph ^= (++rst == NST) ? 1u : 0u, rst = (rst == NST) ? 0 : rst) {
                        if (lane == 0) {
                            const bool ok = mbar_wait_bounded(&empty[rst], rph ^ 1u, p.ctl, 2, abort_flag);
                            const int ce = min(cb + CB, Rg.uhi);
                            const int a0 = max(cb, Rg.jlo), a1 = min(ce, Rg.jhi), b0 = max(cb, Rg.klo), b1 = min(ce, Rg.khi);
                            const uint32_t bj = a1 > a0 ? (uint32_t)(a1 - a0) * kJS * 4u : 0u, bk = b1 > b0 ? (uint32_t)(b1 - b0) * kJS * 4u : 0u;
                            float *st_j = ring + (size_t)rst * 2 * CB * kJS, *st_k = st_j + (size_t)CB * kJS;
                            if (ok) mbar_arrive_expect_tx(&full[rst], bj + bk);
                            if (ok && bj) bulk_g2s(st_j + (size_t)(a0 - cb) * kJS, J + (Rg.jg + (a0 - Rg.jlo)) * kJS, bj, &full[rst]);
                            if (ok && bk) bulk_g2s(st_k + (size_t)(b0 - cb) * kJS, J + (Rg.kg + (b0 - Rg.klo)) * kJS, bk, &full[rst]);
                        }
                        __syncwarp();
                    }
                }
            }
            continue;
        }

        // ---------------- field warps: tables, amplitudes, chain data
        for (int i = tid; i <= sd.ST; i += NCT) s_bo[i] = p.bo[sd.tab_off + i];
        const int rows = N + 2 * APAD;
        const int64_t a0 = sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
        for (int i = tid; i < rows * G; i += NCT) {
            const int ch = i / rows, R = i - ch * rows, x = R - APAD;  // lanes over modes: a chain is contiguous
            amp[R * RS + ch] = (x >= 0 && x < N && ch < gr.count) ? __ldcg(A + a0 + (int64_t)ch * N + x) : f2(0.f, 0.f);
        }
        double E = 0.0;
        float beta = 0.f;
        unsigned n_acc = 0u;
        if (c < gr.count) {
            E = __ldcg(p.E + gr.chain0 + c);
            beta = (float)p.beta[temp];
        }
        named_bar(1, NCT);
        for (int i = tid; i < rows * G; i += NCT) {
            const int R = i / G, ch = i % G;
            const float2 x = amp[R * RS + ch], y = R + 1 < rows ? amp[(R + 1) * RS + ch] : f2(0.f, 0.f);
            win[i] = make_float4(x.x, y.x, x.y, y.y);
        }
        const uint32_t *binfo = p.blkinfo + sd.blk_off;
        const long long tr_at = p.trace ? p.ctl->trace_at : 0ll;  // update trace: absolute sweep + 1 (0 = none)
        const int tr_u = p.trace ? p.ctl->trace_update : -1;
        const float cc = (float)p.cc;

        for (int n = n0; n < n1;) {
            const int sw = n / half, u0 = n - sw * half, u1 = min(half, u0 + n1 - n);
            const uint32_t sweep = (uint32_t)(sweep_base + sw);
            n += u1 - u0;
            // the sweep's pair sequence (every warp has read the previous sweep's last entry before that update's barrier)
            for (int i = tid; i < half; i += NCT) {
                int j, k;
                pair_jk(p.seed, (uint32_t)gr.sample, sweep, (uint32_t)i, N, j, k);
                s_pair[i] = j | (k << 16);
            }
            named_bar(1, NCT);
            for (int u = u0; u < u1; ++u, ++upd) {
                const int jk = s_pair[u], j = jk & 0xffff, k = jk >> 16;
                const Ranges Rg = update_ranges(sd, s_bo, mode_blk, j, k);
                const int buf = (int)(upd & 1u);
                if (C > 1 && tid == 0) mbar_arrive_expect_tx(&pbar[buf], (uint32_t)(C * G * 4));
                PartialsX2 F;
                F.zero();
                for (int cb = Rg.ulo + rank * CB; cb < Rg.uhi; cb += C * CB, ++q, rph ^= (++rst == NST) ? 1u : 0u, rst = (rst == NST) ? 0 : rst) {
                    // a chunk whose copies have landed is processed; a wait that gives up, or sees the abort flag, skips it
                    const bool landed = mbar_wait_bounded(&full[rst], rph, p.ctl, 3, abort_flag);
                    const int b = cb + worker;
                    if (b < Rg.uhi && landed) {
                        const uint32_t info = __ldg(binfo + b);
                        const int s0 = (int)(info >> 16) * TS, x0 = (int)(info & 0xffffu) * TX;
                        const bool inj = b >= Rg.jlo && b < Rg.jhi, ink = b >= Rg.klo && b < Rg.khi;
                        const float *st_j = ring + (size_t)rst * 2 * CB * kJS + (size_t)worker * kJS, *st_k = st_j + (size_t)CB * kJS;
                        if (inj && ink) process_block_x2<G, 3>(amp, win, c, s0, x0, j, k, st_j, st_k, F);
                        else if (inj) process_block_x2<G, 1>(amp, win, c, s0, x0, j, k, st_j, st_k, F);
                        else if (ink) process_block_x2<G, 2>(amp, win, c, s0, x0, j, k, st_j, st_k, F);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[rst]);
                }
                // the update's slot: every lane finishes its chain's proposal, and B_jk = sum_s conj(a_{s-j})
                // J_j[s][{k, s-k}] a_{s-k} over s in [max(j,k), min(j,k) + N) is split over the workers
                const int slot = (int)(bcnt % kBD);
                const uint32_t bph = (bcnt / kBD) & 1u;
                ++bcnt;
                const float2 aj = amp[(j + APAD) * RS + c], ak = amp[(k + APAD) * RS + c];
                Proposal<float> P;
                P.nj = P.aj = aj; P.nk = P.ak = ak; P.U = 1.f;
                if (mbar_wait_bounded(&bfull[slot], bph, p.ctl, 5, abort_flag)) {
                    P = finish_proposal<float>(draws[slot * G + c], aj, ak);
                    const float *bv = bval + slot * p.maxN;
                    const int s_lo = max(j, k), s_hi = min(j, k) + N;
                    for (int s = s_lo + rank * CB + worker; s < s_hi; s += C * CB)
                        caxpy(F.B, bv[s - s_lo], cmulc(amp[(s - j + APAD) * RS + c], amp[(s - k + APAD) * RS + c]));
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&bempty[slot]);
                // this lane's share of Re[conj(dj) h_j + conj(dk) h_k + conj(dj) dk B_jk + conj(dj) conj(dk) A_jk]
                const float hs[8] = {F.hjx.x + F.hjx.y, (F.hjy.x + F.hjy.y) - (F.hjyn.x + F.hjyn.y), F.hkx.x + F.hkx.y,
                                     (F.hky.x + F.hky.y) - (F.hkyn.x + F.hkyn.y), F.B.x, F.B.y, F.A.x, F.A.y};
                const float2 dj = f2(P.nj.x - aj.x, P.nj.y - aj.y), dk = f2(P.nk.x - ak.x, P.nk.y - ak.y);
                float v = dj.x * hs[0] + dj.y * hs[1] + dk.x * hs[2] + dk.y * hs[3];
                v += (dj.x * dk.x + dj.y * dk.y) * hs[4] + (dj.y * dk.x - dj.x * dk.y) * hs[5];
                v += (dj.x * dk.x - dj.y * dk.y) * hs[6] + (dj.x * dk.y + dj.y * dk.x) * hs[7];
#pragma unroll
                for (int o = G; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (wq == 0) part[(buf * NCW + warp) * G + c] = v;
                const bool traced = tr_at == sweep_base + sw + 1 && u == tr_u;
                if (traced) {  // the record's sums, added over the warps in FP64, and the state before the update
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float s = hs[e];
                        for (int o = G; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                        if (wq == 0 && c < gr.count) atomicAdd(p.trace + (int64_t)id * kTraceRec + 2 + e, (double)s);
                    }
                    if (rank == 0)
                        for (int ch = 0; ch < gr.count; ++ch) {
                            const uint32_t cid = __shfl_sync(0xffffffffu, id, ch);
                            double2 *o = reinterpret_cast<double2 *>(p.trace + (int64_t)p.n_chains * kTraceRec) + sd.a_off +
                                         (int64_t)(cid - (uint32_t)sd.chain0) * N;
                            for (int x = lane; x < N; x += 32)
                                if (warp == 0) o[x] = make_double2((double)amp[(x + APAD) * RS + ch].x, (double)amp[(x + APAD) * RS + ch].y);
                        }
                }
                named_bar(1, NCT);
                // decision: every warp adds the shares in the same order, decides alike and writes the same values, so
                // no second barrier is needed before the next update (its barrier keeps the warps within one update)
                float s = 0.f;
                if (C == 1 || warp == 0) {
                    const float *at = part + buf * NCW * G + c;
#pragma unroll
                    for (int w0 = 0; w0 < NCW; w0 += WPW)
                        if (w0 + wq < NCW) s += at[(w0 + wq) * G];
#pragma unroll
                    for (int o = G; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                }
                if constexpr (C > 1) {  // the blocks' shares, to every block of the cluster (its own included)
                    if (warp == 0) {
                        const uint32_t at = smem_u32(xpart + (buf * C + rank) * G + c), bar = smem_u32(&pbar[buf]);
                        for (int r = wq; r < C; r += WPW) send_async(cluster_map(at, r), s, cluster_map(bar, r));
                    }
                    (void)mbar_wait_bounded(&pbar[buf], (upd >> 1) & 1u, p.ctl, 6, abort_flag);
                    s = 0.f;
#pragma unroll
                    for (int r = 0; r < C; ++r) s += xpart[(buf * C + r) * G + c];
                }
                const float dH = -cc * s;
                const bool acc = c < gr.count && metropolis_accept(dH, beta, P.U);
                if (traced && warp == 0 && rank == 0 && wq == 0 && c < gr.count) {
                    double *rec = p.trace + (int64_t)id * kTraceRec;
                    rec[0] = j; rec[1] = k;
                    rec[10] = P.nj.x; rec[11] = P.nj.y; rec[12] = P.nk.x; rec[13] = P.nk.y;
                    rec[14] = P.U; rec[15] = dH; rec[16] = acc ? 1.0 : 0.0; rec[17] = beta; rec[18] = E; rec[19] = 1.0;
                }
                if (acc && wq == 0) {
                    // the window rows j-1, j, k-1, k: row R holds (a_R, a_{R+1}); a neighbour that is the other updated
                    // mode takes its new value (no other amplitude changes in this update)
                    const float2 nj = P.nj, nk = P.nk;
                    float2 *pj = amp + (j + APAD) * RS + c, *pk = amp + (k + APAD) * RS + c;
                    const float2 jm = (j - 1 == k) ? nk : pj[-RS], jp = (j + 1 == k) ? nk : pj[RS];
                    const float2 km = (k - 1 == j) ? nj : pk[-RS], kp = (k + 1 == j) ? nj : pk[RS];
                    *pj = nj; *pk = nk;
                    float4 *wj = win + (j + APAD) * G + c, *wk = win + (k + APAD) * G + c;
                    wj[-G] = make_float4(jm.x, nj.x, jm.y, nj.y);
                    wj[0] = make_float4(nj.x, jp.x, nj.y, jp.y);
                    wk[-G] = make_float4(km.x, nk.x, km.y, nk.y);
                    wk[0] = make_float4(nk.x, kp.x, nk.y, kp.y);
                }
                if (acc && warp == 0) { E += (double)dH; ++n_acc; }
                __syncwarp();
            }
            // interior measurement point: snapshot amplitudes and energies
            const long long done = sweep_base + sw + 1;
            if (u1 == half && p.measure_every > 0 && done % p.measure_every == 0 && sw + 1 < n_sweeps) {
                const int kk = (int)(done / p.measure_every - sweep_base / p.measure_every - 1);
                named_bar(1, NCT);
                if (rank == 0 && kk >= 0 && kk < p.n_snap_max) {
                    float2 *dst = reinterpret_cast<float2 *>(p.snap_a) + (int64_t)kk * p.a_total + a0;
                    for (int i = tid; i < N * gr.count; i += NCT) {
                        const int ch = i / N, x = i - ch * N;
                        dst[i] = amp[(x + APAD) * RS + ch];
                    }
                    if (tid < gr.count) p.snap_E[(int64_t)kk * p.n_chains + gr.chain0 + tid] = E;
                }
                named_bar(1, NCT);
            }
        }
        // ---- write back the group's state and counters
        named_bar(1, NCT);
        if (rank == 0) {
            for (int i = tid; i < N * gr.count; i += NCT) {
                const int ch = i / N, x = i - ch * N;
                __stcg(A + a0 + i, amp[(x + APAD) * RS + ch]);
            }
            if (tid < gr.count) {
                const int slot = gr.chain0 + tid;
                __stcg(p.E + slot, E);
                p.mc_acc[slot] += n_acc;
                p.mc_att[slot] += (unsigned long long)(n1 - n0);
            }
            __threadfence();
            named_bar(1, NCT);
            if (tid == 0) asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p.progress + g), "r"(ci + 1) : "memory");
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

// ------------------------------------------------------------------------------------------------ host launchers
namespace {

size_t smem_limit() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return (size_t)v;
}

// Ring stages for the largest N (0 when fewer than kNstMin fit).
template <int G, int NCW, int C> int comb_stages(int maxN, size_t limit) {
    int d = kNstMax;
    while (d >= kNstMin && comb_smem<G, NCW, C>(maxN, d).total > limit) --d;
    return d >= kNstMin ? d : 0;
}

template <int G, int NCW, int C> cudaError_t launch_comb_t(const SweepParams &p, int clusters, cudaStream_t s) {
    SweepParams q = p;
    q.nst = comb_stages<G, NCW, C>(p.maxN, smem_limit());
    if (q.nst == 0) return cudaErrorInvalidConfiguration;
    const size_t sm = comb_smem<G, NCW, C>(p.maxN, q.nst).total;
    auto *k = comb_sweep_kernel<G, NCW, C>;
    // the kernel's largest limit, not this context's: contexts of other sizes launch it too
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit());
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * C);
    cfg.blockDim = dim3((NCW + 1) * 32);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, q);
}

// Clusters the device holds at once (0: the shape does not fit).
template <int G, int NCW, int C> int comb_clusters_t(int maxN, int sms) {
    const int d = comb_stages<G, NCW, C>(maxN, smem_limit());
    if (d == 0) return 0;
    const size_t sm = comb_smem<G, NCW, C>(maxN, d).total;
    auto *k = comb_sweep_kernel<G, NCW, C>;
    int nb = 0;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit());
    if (e == cudaSuccess && C == 1) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, (NCW + 1) * 32, sm);
        nb *= sms;
    } else if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3((NCW + 1) * 32);
        cfg.dynamicSmemBytes = sm;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&nb, k, &cfg);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return nb;
}

}  // namespace

#define PT_COMB_VARIANTS(X)                                      \
    X(8, 7, 1) X(8, 11, 1) X(8, 15, 1)                           \
    X(16, 7, 1) X(16, 11, 1) X(16, 15, 1)                        \
    X(32, 3, 1) X(32, 7, 1) X(32, 9, 1) X(32, 11, 1)             \
    X(8, 11, 2) X(8, 11, 4) X(8, 11, 8) X(8, 7, 2) X(8, 7, 4) X(8, 7, 8)

bool comb_variant_exists(int G, int ncw, int cl) {
#define X(g, n, cc) if (G == g && ncw == n && cl == cc) return true;
    PT_COMB_VARIANTS(X)
#undef X
    return false;
}

cudaError_t launch_comb(int G, int ncw, int cl, const SweepParams &p, int clusters, cudaStream_t s) {
#define X(g, n, cc) if (G == g && ncw == n && cl == cc) return launch_comb_t<g, n, cc>(p, clusters, s);
    PT_COMB_VARIANTS(X)
#undef X
    return cudaErrorInvalidValue;
}

int comb_clusters(int G, int ncw, int cl, int maxN, int sms) {
#define X(g, n, cc) if (G == g && ncw == n && cl == cc) return comb_clusters_t<g, n, cc>(maxN, sms);
    PT_COMB_VARIANTS(X)
#undef X
    return 0;
}

}  // namespace ptgb
