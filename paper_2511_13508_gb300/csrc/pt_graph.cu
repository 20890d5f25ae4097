// pt_graph.cu -- FP32 sweep and energy kernels for explicit interaction lists (the random-frequency
// mode-locked graph of arXiv 2511.13508, Sec. II.C, or any list of quadruplets).
//
// Three sweeps, by the number of records of an update and N (graph_variant below): one chain per block of two warps for
// few records, a table of pair products shared by the records of a dense graph, and, for the rest and for the energies,
// one thread block per group of up to 8 chains of one disorder sample.  In that last one a lane is (chain c, worker w):
// the 128 workers of the block split the quadruplets that hold the updated modes j or k, and the 8
// lanes of a worker read each incidence record once for their 8 chains.  An incidence record of mode l
// is (the other three modes in position order, (q << 2) | position of l) with its coupling alongside,
// so a lane needs no search and no dependent load to evaluate a quadruplet.  Per chain the lane
// accumulates the local fields of j and k and the j-k cross term (Sec. III.A.1 and III.A.3; term of
// quadruplet (q0, q1, q2, q3): -cc J Re(conj(a_q0) a_q1 a_q2 conj(a_q3))):
//     h_l = sum_{q holding l} J_q (product of the other three factors), conjugated when l sits at
//           position 1 or 2, so that H = -cc Re(conj(a_l) h_l) + (terms without l);
//     dH  = -cc Re[ conj(dj) h_j + conj(dk) h_k + sum_{q holding j and k} J_q x x dxj dxk ],
// with dxl = conj(dl) at positions 0 and 3, dl at 1 and 2.  Products in FP32, energies in FP64.
#include <cstdint>
#include "pt_bulk.cuh"
#include "pt_common.cuh"
#include "pt_kernels.h"
#include "pt_move.cuh"

namespace ptgb {

namespace {

constexpr int kGG = 8;                      // chains per block
constexpr int kGThreads = 1024;             // 32 warps
constexpr int kGWarps = kGThreads / 32;
constexpr int kGWorkers = kGThreads / kGG;  // 128
// row stride of the amplitude table (float2), unpadded: a warp's four records then gather from two 64-byte halves
// of the banks instead of windows at 16 offsets (fewer bank conflicts; measured on GB300, random graph N = 64:
// 4.46M -> 4.73M chain-sweeps/s against a stride of kGG + 1)
constexpr int kGRS = kGraphRowStride;
static_assert(kGRS == kGG, "row stride");

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// factor of position p in the term: conjugated at positions 0 and 3
__device__ __forceinline__ float2 fac(float2 v, int p) { return (p == 0 || p == 3) ? make_float2(v.x, -v.y) : v; }

struct GraphProposal {
    float2 dj, dk, nj, nk;
    float U;
};

__device__ __forceinline__ GraphProposal graph_proposal(uint64_t seed, uint32_t chain_id, uint32_t sweep,
                                                        uint32_t update, float2 aj, float2 ak) {
    // the pair move of Sec. III.A.1: K^4 = |a_j|^4 + |a_k|^4, theta ~ U[0, pi/2], fresh uniform phases;
    // mode j receives K sqrt(cos theta), mode k receives K sqrt(sin theta)
    GraphProposal P;
    const u32x4 w = draw(seed, chain_id, sweep, update, kTagPropose);
    const float uj = aj.x * aj.x + aj.y * aj.y, uk = ak.x * ak.x + ak.y * ak.y;
    const float K = sqrtf(sqrtf(uj * uj + uk * uk));
    const float kInv = 2.3283064365386963e-10f;
    const float fj = ((float)w.x + 0.5f) * kInv, fk = ((float)w.y + 0.5f) * kInv, ft = ((float)w.z + 0.5f) * kInv;
    float sj, cj, sk, ck, st, ct;
    sincospif(2.0f * fj, &sj, &cj);
    sincospif(2.0f * fk, &sk, &ck);
    sincospif(0.5f * ft, &st, &ct);
    const float Aj = K * sqrtf(ct), Ak = K * sqrtf(st);
    P.nj = make_float2(Aj * cj, Aj * sj);
    P.nk = make_float2(Ak * ck, Ak * sk);
    P.dj = make_float2(P.nj.x - aj.x, P.nj.y - aj.y);
    P.dk = make_float2(P.nk.x - ak.x, P.nk.y - ak.y);
    P.U = ((float)w.w + 0.5f) * kInv;
    return P;
}

}  // namespace

// Variants by how an update's records reach the workers:
//  kPlain: each worker loads its records from global memory (L2) as it goes (the largest graphs).
//  kStage: the two lists fit in shared memory; the whole block copies them there with asynchronous copies
//    while the leaders draw the proposal (one L2 latency per update instead of one per record and worker).
//  kWarp (graph_warp_kernel): few records per update (sparse graphs, small N), one chain per block of two warps.
//  kTable (graph_table_kernel): pair products of 8 or 4 chains in shared memory (dense graphs of small N).
enum GraphVariant : int { kPlain = 0, kStage = 2, kWarp = 3, kTable = 4 };

// Shared-memory layout of the sweep kernel: amplitudes [maxN][kGRS] float2, record offsets [maxN + 1] int,
// then (kStage) the staged records [cap] int4 and couplings [cap] float.
struct GraphSmem {
    size_t inc, rec, J, total;
};
__host__ __device__ inline GraphSmem graph_smem(int maxN, int cap) {
    GraphSmem g;
    g.inc = (size_t)maxN * kGRS * sizeof(float2);
    g.rec = (g.inc + (size_t)(maxN + 1) * sizeof(int) + 15) / 16 * 16;
    g.J = g.rec + (size_t)cap * sizeof(int4);
    g.total = g.J + (size_t)cap * sizeof(float);
    return g;
}

template <int kVar>
__global__ void __launch_bounds__(kGThreads) graph_sweep_kernel(GraphParams p) {
    constexpr bool kStageV = kVar == kStage;
    extern __shared__ __align__(16) float2 ga[];  // laid out as graph_smem
    __shared__ float red[kGWarps][kGG][5];
    __shared__ GraphProposal prop[kGG];
    const GroupDev gr = p.groups[blockIdx.x];
    const SampleDev sd = p.samples[gr.sample];
    const int N = sd.N, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int c = lane % kGG, worker = warp * (32 / kGG) + lane / kGG;
    const bool leader = tid < kGG;  // warp 0, worker 0: chain c = tid
    float2 *A = p.a + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
    for (int i = tid; i < N * kGG; i += kGThreads) {
        const int x = i / kGG, cc = i % kGG;
        ga[x * kGRS + cc] = cc < gr.count ? A[(int64_t)cc * N + x] : make_float2(0.f, 0.f);
    }
    double E = 0.0;
    float beta = 0.f;
    uint32_t cid = 0;
    unsigned long long acc = 0, att = 0;
    if (leader && c < gr.count) {
        const int slot = gr.chain0 + c;
        const int r = (slot - sd.chain0) / p.nT, t = p.label[slot];
        E = p.E[slot];
        beta = (float)p.beta[t];
        cid = (uint32_t)((gr.sample * p.R + r) * p.nT + t);
    }
    const int cap = 2 * p.max_deg;
    const GraphSmem lay = graph_smem(p.maxN, kStageV ? cap : 0);
    unsigned char *sbase = reinterpret_cast<unsigned char *>(ga);
    int *inc_off_s = reinterpret_cast<int *>(sbase + lay.inc);
    int4 *rec_s = reinterpret_cast<int4 *>(sbase + lay.rec);
    float *recJ_s = reinterpret_cast<float *>(sbase + lay.J);
    if (kStageV)
        for (int i = tid; i <= N; i += kGThreads) inc_off_s[i] = p.inc_off[sd.mode_off + i];
    const int *inc_off = kStageV ? inc_off_s : p.inc_off + sd.mode_off;
    const int4 *rec = p.rec + sd.inc_off;
    const float *recJ = p.recJ + sd.inc_off;
    const float cc_f = (float)p.cc;
    const long long base = p.ctl->sweep_base;
    // update trace: absolute sweep + 1 and update to record (0 = none)
    const long long tr_at = p.trace ? p.ctl->trace_at : 0ll;
    const int tr_u = p.trace ? p.ctl->trace_update : -1;
    __syncthreads();
    for (int sw = 0; sw < p.n_sweeps; ++sw) {
        const uint32_t sweep = (uint32_t)(base + sw);
        for (int u = 0; u < N / 2; ++u) {
            int j, k;
            pair_jk(p.seed, (uint32_t)gr.sample, sweep, (uint32_t)u, N, j, k);
            if (kStageV) {  // the update's records into shared memory (the previous update's reads are done)
                const int oj = inc_off[j], nj = inc_off[j + 1] - oj, ok = inc_off[k], nk = inc_off[k + 1] - ok;
                for (int i = tid; i < nj + nk; i += kGThreads) {
                    const int r = i < nj ? oj + i : ok + i - nj;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(rec_s + i)), "l"(rec + r)
                                 : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(recJ_s + i)), "l"(recJ + r)
                                 : "memory");
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            if (leader) prop[c] = graph_proposal(p.seed, cid, sweep, (uint32_t)u, ga[j * kGRS + c], ga[k * kGRS + c]);
            if (kStageV) asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            const GraphProposal P = prop[c];
            float2 hj = make_float2(0.f, 0.f), hk = make_float2(0.f, 0.f);
            float cr = 0.f;
            const int oj = inc_off[j], nj = inc_off[j + 1] - oj;
            const int ok = inc_off[k], nk = inc_off[k + 1] - ok;
            // one record of mode j (onj) or k: its field term, and for a quadruplet holding both (counted once,
            // from j's list) k's term and the cross term
            auto term = [&](const int4 R4, const float J, const bool onj) {
                const int pos = R4.w & 3;              // position of the record's own mode (j or k)
                const int otherR = (onj ? k : j) * kGRS;  // the other updated mode, possibly among the three
                const int o[3] = {R4.x, R4.y, R4.z};   // row offsets of A, B, C
                int po = -1;                           // index (0..2) of the other updated mode among them
#pragma unroll
                for (int m = 0; m < 3; ++m) if (o[m] == otherR) po = m;
                if (!onj && po >= 0) return;
                const float2 fa = ga[o[0] + c], fb = ga[o[1] + c], fc = ga[o[2] + c];
                // field of the record's mode: J a_A a_B conj(a_C)
                const float2 ab = cmulf(fa, fb);
                const float2 X = make_float2(J * (ab.x * fc.x + ab.y * fc.y), J * (ab.y * fc.x - ab.x * fc.y));
                if (onj) { hj.x += X.x; hj.y += X.y; } else { hk.x += X.x; hk.y += X.y; }
                if (onj && po >= 0) {
                    // the quadruplet holds j (this record) and k: k's field and the cross term, from the
                    // positions of the factors (conjugated at positions 0 and 3)
                    const int opos[3] = {(R4.w >> 2) & 3, (R4.w >> 4) & 3, (R4.w >> 6) & 3};
                    const float2 f[3] = {fac(fa, opos[0]), fac(fb, opos[1]), fac(fc, opos[2])};
                    const float2 own = fac(ga[j * kGRS + c], pos);
                    const int pk = opos[po];
                    float2 Y = make_float2(J * own.x, J * own.y), Z = make_float2(J, 0.f);
#pragma unroll
                    for (int m = 0; m < 3; ++m)
                        if (m != po) { Y = cmulf(Y, f[m]); Z = cmulf(Z, f[m]); }
                    if (pk == 1 || pk == 2) Y.y = -Y.y;
                    hk.x += Y.x; hk.y += Y.y;
                    const float2 dxj = (pos == 0 || pos == 3) ? make_float2(P.dj.x, -P.dj.y) : P.dj;
                    const float2 dxk = (pk == 0 || pk == 3) ? make_float2(P.dk.x, -P.dk.y) : P.dk;
                    cr += cmulf(Z, cmulf(dxj, dxk)).x;
                }
            };
            {   // j's list, then k's (the list a record comes from is then known at compile time)
                for (int idx = worker; idx < nj; idx += kGWorkers)
                    term(kStageV ? rec_s[idx] : __ldg(rec + oj + idx), kStageV ? recJ_s[idx] : __ldg(recJ + oj + idx),
                         true);
                for (int idx = worker; idx < nk; idx += kGWorkers)
                    term(kStageV ? rec_s[nj + idx] : __ldg(rec + ok + idx),
                         kStageV ? recJ_s[nj + idx] : __ldg(recJ + ok + idx), false);
            }
            // reduce over the 4 workers of the warp, then over the warps in a fixed order
            float v[5] = {hj.x, hj.y, hk.x, hk.y, cr};
#pragma unroll
            for (int o = kGG; o < 32; o <<= 1)
#pragma unroll
                for (int e = 0; e < 5; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
            if (lane < kGG) {
#pragma unroll
                for (int e = 0; e < 5; ++e) red[warp][c][e] = v[e];
            }
            __syncthreads();
            if (leader && c < gr.count) {
                float t[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
                for (int w = 0; w < kGWarps; ++w)
#pragma unroll
                    for (int e = 0; e < 5; ++e) t[e] += red[w][c][e];
                // Re(conj(d) h) = d.x h.x + d.y h.y
                const float dH = -cc_f * (P.dj.x * t[0] + P.dj.y * t[1] + P.dk.x * t[2] + P.dk.y * t[3] + t[4]);
                ++att;
                const bool accept = dH <= 0.f || P.U < expf(-beta * dH);
                if (tr_at == base + sw + 1 && u == tr_u) {
                    // the record of this update and the chain's state before it (this leader is the only writer
                    // of its chain's column, so the table still holds the old a_j, a_k)
                    double *rec_o = p.trace + (int64_t)cid * kTraceRec;
                    const double v[kTraceRec] = {(double)j, (double)k, (double)t[0], (double)t[1], (double)t[2],
                                                 (double)t[3], (double)t[4], 0.0, 0.0, 0.0, (double)P.nj.x,
                                                 (double)P.nj.y, (double)P.nk.x, (double)P.nk.y, (double)P.U,
                                                 (double)dH, accept ? 1.0 : 0.0, (double)beta, E, 1.0};
                    for (int e = 0; e < kTraceRec; ++e) rec_o[e] = v[e];
                    double2 *st_o = reinterpret_cast<double2 *>(p.trace + (int64_t)p.n_chains * kTraceRec) + sd.a_off +
                                    (int64_t)(cid - (uint32_t)sd.chain0) * N;
                    for (int x = 0; x < N; ++x) {
                        const float2 a = ga[x * kGRS + c];
                        st_o[x] = make_double2((double)a.x, (double)a.y);
                    }
                }
                if (accept) {
                    ga[j * kGRS + c] = P.nj;
                    ga[k * kGRS + c] = P.nk;
                    E += (double)dH;
                    ++acc;
                }
            }
            // the leaders' amplitude writes are ordered before every read of the next update by the
            // barrier after its proposals
        }
        const long long done = base + sw + 1;
        if (p.measure_every > 0 && done % p.measure_every == 0 && sw + 1 < p.n_sweeps) {
            __syncthreads();
            const int kk = (int)(done / p.measure_every - base / p.measure_every - 1);
            if (kk >= 0 && kk < p.n_snap_max) {
                float2 *dst = p.snap_a + (int64_t)kk * p.a_total + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
                for (int i = tid; i < N * gr.count; i += kGThreads) {
                    const int cc = i / N, x = i % N;
                    dst[(int64_t)cc * N + x] = ga[x * kGRS + cc];
                }
                if (leader && c < gr.count) p.snap_E[(int64_t)kk * p.n_chains + gr.chain0 + c] = E;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    for (int i = tid; i < N * gr.count; i += kGThreads) {
        const int cc = i / N, x = i % N;
        A[(int64_t)cc * N + x] = ga[x * kGRS + cc];
    }
    if (leader && c < gr.count) {
        const int slot = gr.chain0 + c;
        if (!isfinite(E)) record_error(p.ctl, kErrNaN, 30);
        p.E[slot] = E;
        p.mc_acc[slot] += acc;
        p.mc_att[slot] += att;
    }
}

// ------------------------------------------------------------------------------------------------
// One chain per block of two warps, for updates of few records.  Such an update is bound by its chain of latencies (with a
// block of 8 chains and its two barriers 1.94 us at N = 2048, z = 16; with one warp doing everything 0.69 us).  The
// field warp spreads the records over its lanes, reduces one value, decides and writes; everything else is the helper's,
// an update or more ahead: pairs, record ranges and random numbers of 32 updates at once (a lane each), the records of
// the next kWarpAhead updates on their way into shared memory, and the next proposal, scaled for both outcomes of the
// current update.  One barrier per update.
// dH = Re[conj(dj) h_j] with a_k already replaced + Re[conj(dk) h_k] with a_j not yet replaced (times -cc), so that
// quadruplets holding both modes need no cross term.
constexpr int kWarpRec = 64;   // records per update that are copied ahead (further ones load as they go)
constexpr int kWarpAhead = 4;  // updates ahead

struct WarpDraw {  // one update: pair, record ranges and the random part of the proposal
    int jk, oj, nj, ok, nk, pad[3];
    ProposalDraw<float> D;
};
struct WarpProposal {
    float2 aj, ak, nj, nk;  // old and proposed amplitudes
    float U, pad[3];
};

__global__ void __launch_bounds__(64, 10) graph_warp_kernel(GraphParams p) {
    extern __shared__ __align__(16) float2 wa[];  // [N]
    __shared__ WarpDraw dr[64];                   // two batches of 32 updates
    __shared__ int4 ring[kWarpAhead][kWarpRec];
    __shared__ float ringJ[kWarpAhead][kWarpRec];
    __shared__ WarpProposal prop[2][2];           // [update & 1][previous update accepted]
    __shared__ int s_ok[2];                       // outcome of update n at [n & 1]
    const int lane = threadIdx.x & 31, slot = blockIdx.x;
    const bool helper = threadIdx.x >= 32;
    const int si = p.chain_sample[slot];
    const SampleDev sd = p.samples[si];
    const int N = sd.N, half = N / 2, total = p.n_sweeps * half;
    float2 *A = p.a + sd.a_off + (int64_t)(slot - sd.chain0) * N;
    for (int x = threadIdx.x; x < N; x += 64) wa[x] = A[x];
    const int t = p.label[slot];
    const uint32_t cid = (uint32_t)((si * p.R + (slot - sd.chain0) / p.nT) * p.nT + t);
    const float beta = (float)p.beta[t], cc = (float)p.cc;
    double E = p.E[slot];
    unsigned n_acc = 0u;
    const int4 *rec = p.rec + sd.inc_off;
    const float *recJ = p.recJ + sd.inc_off;
    const long long base = p.ctl->sweep_base;
    const long long tr_at = p.trace ? p.ctl->trace_at : 0ll;
    const int tr_u = p.trace ? p.ctl->trace_update : -1;
    auto draw_batch = [&](int n0) {
        const int n = n0 + lane;
        if (n < total) {
            const int sw = n / half, u = n - sw * half;
            const int *inc_off = p.inc_off + sd.mode_off;
            WarpDraw &w = dr[n & 63];
            int j, k;
            pair_jk(p.seed, (uint32_t)si, (uint32_t)(base + sw), (uint32_t)u, N, j, k);
            w.jk = j | (k << 16);
            w.oj = __ldg(inc_off + j); w.nj = __ldg(inc_off + j + 1) - w.oj;
            w.ok = __ldg(inc_off + k); w.nk = __ldg(inc_off + k + 1) - w.ok;
            w.D = draw_proposal<float>(p.seed, cid, (uint32_t)(base + sw), (uint32_t)u);
        }
        __syncwarp();
    };
    auto prefetch = [&](int n) {  // one copy group per update, empty past the end
        if (n < total) {
            const WarpDraw &w = dr[n & 63];
            const int s = n % kWarpAhead, nj = w.nj, nr = nj + w.nk, kofs = w.ok - nj, jofs = w.oj;
#pragma unroll
            for (int e = 0; e < kWarpRec / 32; ++e) {
                const int i = lane + 32 * e;
                if (i < nr) {
                    const int r = (i < nj ? jofs : kofs) + i;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(&ring[s][i])), "l"(rec + r) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(&ringJ[s][i])), "l"(recJ + r) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // proposal of update n after update n - 1 with proposal Q was rejected (lane 0) or accepted (lane 1); only modes of
    // update n - 1 may be written meanwhile, and their values are taken from Q
    auto propose = [&](int n, int jkq, const WarpProposal *Q) {
        const WarpDraw &w = dr[n & 63];
        const int j = w.jk & 0xffff, k = w.jk >> 16;
        float2 aj = wa[j], ak = wa[k];
        if (Q) {
            const int jq = jkq & 0xffff, kq = jkq >> 16;
            const float2 qj = lane ? Q->nj : Q->aj, qk = lane ? Q->nk : Q->ak;
            if (j == jq) aj = qj; else if (j == kq) aj = qk;
            if (k == jq) ak = qj; else if (k == kq) ak = qk;
        }
        const Proposal<float> P = finish_proposal<float>(w.D, aj, ak);
        WarpProposal &o = prop[n & 1][lane];
        o.aj = aj; o.ak = ak; o.nj = P.nj; o.nk = P.nk; o.U = P.U;
    };
    if (helper) {
        draw_batch(0);
        for (int n = 0; n < kWarpAhead; ++n) prefetch(n);
        asm volatile("cp.async.wait_group %0;" ::"n"(kWarpAhead - 1) : "memory");
    }
    __syncthreads();
    if (helper && lane < 2 && total > 0) propose(0, 0, nullptr);
    if (threadIdx.x < 2) s_ok[threadIdx.x] = 0;
    __syncthreads();
    int sw = 0, u = 0;
    for (int n = 0; n < total; ++n) {
        const int at = n & 63;
        const WarpProposal &P = prop[n & 1][s_ok[(n & 1) ^ 1]];
        if (helper) {
            const int jk = dr[at].jk;
            if ((n & 31) == 0) draw_batch(n + 32);
            if (lane < 2 && n + 1 < total) propose(n + 1, jk, &P);
            // update n + 1's records are complete when only the later groups are in flight; the slot of update n is
            // free for update n + kWarpAhead after the barrier
            asm volatile("cp.async.wait_group %0;" ::"n"(kWarpAhead - 2) : "memory");
        } else {
            const int jk = dr[at].jk, j = jk & 0xffff, k = jk >> 16, nj = dr[at].nj, nr = nj + dr[at].nk;
            const bool traced = tr_at == base + sw + 1 && u == tr_u;
            const float2 njv = P.nj, nkv = P.nk;
            const float2 dj = make_float2(njv.x - P.aj.x, njv.y - P.aj.y), dk = make_float2(nkv.x - P.ak.x, nkv.y - P.ak.y);
            // field term J a_A a_B conj(a_C) of a record's mode (row offsets are modes x the group kernels' table stride),
            // with a_k replaced in the records of j, as its share of Re[conj(d) h]
            auto term = [&](const int4 R4, const float J, const bool onj) {
                const int a_ = R4.x / kGraphRowStride, b_ = R4.y / kGraphRowStride, c_ = R4.z / kGraphRowStride;
                float2 fa = wa[a_], fb = wa[b_], fc = wa[c_];
                if (onj && a_ == k) fa = nkv;
                if (onj && b_ == k) fb = nkv;
                if (onj && c_ == k) fc = nkv;
                const float2 d = onj ? dj : dk, ab = cmulf(fa, fb);
                return J * (d.x * (ab.x * fc.x + ab.y * fc.y) + d.y * (ab.y * fc.x - ab.x * fc.y));
            };
            auto record = [&](int i, int4 &R4, float &J) {
                if (i < kWarpRec) {
                    R4 = ring[n % kWarpAhead][i];
                    J = ringJ[n % kWarpAhead][i];
                } else {
                    const int r = i < nj ? dr[at].oj + i : dr[at].ok + i - nj;
                    R4 = __ldg(rec + r);
                    J = __ldg(recJ + r);
                }
            };
            float share = 0.f;
            if (nr <= 32) {
                if (lane < nr) share = term(ring[n % kWarpAhead][lane], ringJ[n % kWarpAhead][lane], lane < nj);
            } else {
                // the first two of a lane together, so that their latencies overlap
                int4 r0 = ring[n % kWarpAhead][lane], r1 = make_int4(0, 0, 0, 0);
                const float j0 = ringJ[n % kWarpAhead][lane];
                float j1 = 0.f;
                const int i1 = lane + 32;
                if (i1 < nr) { r1 = ring[n % kWarpAhead][i1]; j1 = ringJ[n % kWarpAhead][i1]; }
                share = term(r0, j0, lane < nj) + term(r1, j1, i1 < nj);
                for (int i = lane + 64; i < nr; i += 32) {
                    int4 R4;
                    float J;
                    record(i, R4, J);
                    share += term(R4, J, i < nj);
                }
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) share += __shfl_xor_sync(0xffffffffu, share, o);
            const float dH = -cc * share;
            const bool acc = metropolis_accept(dH, beta, P.U);
            if (traced) {
                // the sums of the record: h_j, h_k, and the part of dH bilinear in dj and dk
                float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
                for (int i = lane; i < nr; i += 32) {
                    int4 R4;
                    float J;
                    record(i, R4, J);
                    const int a_ = R4.x / kGraphRowStride, b_ = R4.y / kGraphRowStride, c_ = R4.z / kGraphRowStride;
                    const float2 fa = wa[a_], fb = wa[b_], fc = wa[c_], ab = cmulf(fa, fb);
                    const bool onj = i < nj;
                    v[onj ? 0 : 2] += J * (ab.x * fc.x + ab.y * fc.y);
                    v[onj ? 1 : 3] += J * (ab.y * fc.x - ab.x * fc.y);
                    if (onj && (a_ == k || b_ == k || c_ == k)) {  // the term is linear in a_k or its conjugate
                        const float2 ga = a_ == k ? dk : fa, gb = b_ == k ? dk : fb, gc = c_ == k ? dk : fc, gab = cmulf(ga, gb);
                        v[4] += J * (dj.x * (gab.x * gc.x + gab.y * gc.y) + dj.y * (gab.y * gc.x - gab.x * gc.y));
                    }
                }
#pragma unroll
                for (int e = 0; e < 5; ++e)
                    for (int o = 16; o; o >>= 1) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
                if (lane == 0) {
                    double *out = p.trace + (int64_t)cid * kTraceRec;
                    const double q[kTraceRec] = {(double)j, (double)k, (double)v[0], (double)v[1], (double)v[2], (double)v[3],
                                                 (double)v[4], 0.0, 0.0, 0.0, (double)njv.x, (double)njv.y, (double)nkv.x,
                                                 (double)nkv.y, (double)P.U, (double)dH, acc ? 1.0 : 0.0, (double)beta, E, 1.0};
                    for (int e = 0; e < kTraceRec; ++e) out[e] = q[e];
                }
                double2 *st = reinterpret_cast<double2 *>(p.trace + (int64_t)p.n_chains * kTraceRec) + sd.a_off +
                              (int64_t)(cid - (uint32_t)sd.chain0) * N;
                for (int x = lane; x < N; x += 32) st[x] = make_double2((double)wa[x].x, (double)wa[x].y);
            }
            __syncwarp();  // every lane has read the amplitudes
            if (lane == 0) {
                s_ok[n & 1] = acc ? 1 : 0;
                if (acc) {
                    wa[j] = njv;
                    wa[k] = nkv;
                    E += (double)dH;
                    ++n_acc;
                }
            }
        }
        __syncthreads();
        if (helper) prefetch(n + kWarpAhead);
        if (++u == half) {
            u = 0; ++sw;
            const long long done = base + sw;
            if (p.measure_every > 0 && done % p.measure_every == 0 && sw < p.n_sweeps) {
                const int kk = (int)(done / p.measure_every - base / p.measure_every - 1);
                if (kk >= 0 && kk < p.n_snap_max) {
                    float2 *dst = p.snap_a + (int64_t)kk * p.a_total + sd.a_off + (int64_t)(slot - sd.chain0) * N;
                    for (int x = threadIdx.x; x < N; x += 64) dst[x] = wa[x];
                    if (threadIdx.x == 0) p.snap_E[(int64_t)kk * p.n_chains + slot] = E;
                }
                __syncthreads();
            }
        }
    }
    for (int x = threadIdx.x; x < N; x += 64) A[x] = wa[x];
    if (threadIdx.x == 0) {
        if (!isfinite(E)) record_error(p.ctl, kErrNaN, 30);
        p.E[slot] = E;
        p.mc_acc[slot] += n_acc;
        p.mc_att[slot] += (unsigned long long)total;
    }
}

// ------------------------------------------------------------------------------------------------
// Pair-table sweep, for dense graphs of small N.  The field of mode l is closed partner by partner,
//     h_l = sum_C conj(a_C) sum_{records of l with partner C} J a_A a_B,
// and the products a_A a_B of all N (N-1)/2 pairs stay in shared memory for GC chains: a record is one gather and two
// multiply-adds instead of three gathers and two complex products.  Records come in chunks of four of one mode and one
// partner (graph_chunks on the host); an update's two chunk lists, and the list of the quadruplets that hold both modes
// (for the cross term), are copied into shared memory in bulk.  An accepted update rewrites the 2N - 3 products that hold
// j or k.  The field warps share the chunks; the last warp draws random numbers, scales the next proposal for both
// outcomes of the current update and issues the copies.
// Shared-memory bandwidth bounds it: 17.5 wavefronts per four records of 4 workers x 8 chains, 11 of them gathers.  GB300,
// N = 64 (1260 records per mode), 1024 chains: 226 us per sweep with three gathers per record (graph_sweep_kernel), 108.7
// here; N = 32 59 -> 32.5, N = 96 (4 chains per block) 626 -> 382.

struct TabSmem {
    size_t amp, choff, list, cross, part, draws, prop, ints, total, list_bytes, cross_bytes;
};
__host__ __device__ inline TabSmem tab_smem(int GC, int FW, int N, int max_chunks, int max_cross, int nbuf) {
    TabSmem m;
    size_t o = (size_t)N * (N - 1) / 2 * GC * sizeof(float2);
    auto take = [&](size_t bytes) { const size_t at = (o + 15) / 16 * 16; o = at + bytes; return at; };
    m.amp = take((size_t)N * GC * sizeof(float2));
    m.choff = take((size_t)(N + 1) * sizeof(int));
    m.list_bytes = (size_t)2 * max_chunks * 2 * sizeof(int4);
    m.cross_bytes = (size_t)max_cross * sizeof(int4);
    m.list = take(nbuf * m.list_bytes);
    m.cross = take(nbuf * m.cross_bytes);
    m.part = take((size_t)2 * FW * GC * sizeof(float));
    m.draws = take((size_t)64 * sizeof(ProposalDraw<float>));
    m.prop = take((size_t)4 * GC * sizeof(WarpProposal));
    m.ints = take((size_t)(64 + 2 + 2 + 4) * sizeof(int));
    m.total = o;
    return m;
}

__device__ __forceinline__ int tri_index(int x, int y, int N) {  // pair {x, y}
    const int lo = min(x, y), hi = max(x, y);
    return lo * (2 * N - lo - 1) / 2 + hi - lo - 1;
}
// fused multiply-adds written out: formed again after each accepted update, and at the start of each launch
__device__ __forceinline__ float2 tab_product(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}

template <int GC, int NT>
__global__ void __launch_bounds__(NT, 1) graph_table_kernel(GraphParams p) {
    constexpr int FW = NT / 32 - 1;
    constexpr int WPW = 32 / GC, NWK = FW * WPW, UB = 32 / GC;  // workers per warp, workers, updates drawn at once
    extern __shared__ __align__(16) unsigned char smem[];
    const int nbuf = p.tab_nbuf;
    const TabSmem lay = tab_smem(GC, FW, p.maxN, p.max_chunks, p.max_cross, nbuf);
    float2 *pp = reinterpret_cast<float2 *>(smem), *amp = reinterpret_cast<float2 *>(smem + lay.amp);
    int *choff = reinterpret_cast<int *>(smem + lay.choff);
    float *part = reinterpret_cast<float *>(smem + lay.part);                                // [2][FW][GC]
    ProposalDraw<float> *draws = reinterpret_cast<ProposalDraw<float> *>(smem + lay.draws);  // [2][UB][GC]
    WarpProposal *prop = reinterpret_cast<WarpProposal *>(smem + lay.prop);                  // [2][2][GC]
    int *pairs = reinterpret_cast<int *>(smem + lay.ints);                                   // [64]
    volatile int *s_nx = pairs + 64, *abort_flag = pairs + 66;
    __shared__ uint64_t lbar[2];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c = lane % GC, wq = lane / GC;
    const bool helper = warp == FW;
    const int worker = warp * WPW + wq;
    constexpr int SPLIT = kGG / GC;  // blocks per group of 8
    GroupDev gr = p.groups[blockIdx.x / SPLIT];
    gr.chain0 += (int)(blockIdx.x % SPLIT) * GC;
    gr.count = min(GC, gr.count - (int)(blockIdx.x % SPLIT) * GC);
    if (gr.count <= 0) return;
    const SampleDev sd = p.samples[gr.sample];
    const int N = sd.N, half = N / 2, total = p.n_sweeps * half;
    float2 *A = p.a + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
    if (tid == 0) {
        mbar_init(&lbar[0], 1); mbar_init(&lbar[1], 1);
        *abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = tid; i < N * GC; i += NT) {
        const int ch = i / N, x = i - ch * N;
        amp[x * GC + ch] = ch < gr.count ? A[(int64_t)ch * N + x] : make_float2(0.f, 0.f);
    }
    for (int i = tid; i <= N; i += NT) choff[i] = p.choff[sd.mode_off + i];
    double E = 0.0;
    float beta = 0.f;
    uint32_t cid = 0u;
    unsigned n_acc = 0u;
    if (c < gr.count) {
        const int slot = gr.chain0 + c, t = p.label[slot];
        E = p.E[slot];
        beta = (float)p.beta[t];
        cid = (uint32_t)((gr.sample * p.R + (slot - sd.chain0) / p.nT) * p.nT + t);
    }
    const int4 *chunks = p.chunks + 2 * sd.chunk_off, *cross = p.cross + sd.cross_off;
    const int *xoff = p.xoff + sd.xoff_off;
    const long long base = p.ctl->sweep_base;
    const float cc = (float)p.cc;
    const long long tr_at = p.trace ? p.ctl->trace_at : 0ll;
    const int tr_u = p.trace ? p.ctl->trace_update : -1;
    __syncthreads();
    for (int i = tid; i < N * N * GC; i += NT) {
        const int ch = i % GC, xy = i / GC, x = xy / N, y = xy - x * N;
        if (x < y) pp[tri_index(x, y, N) * GC + ch] = tab_product(amp[x * GC + ch], amp[y * GC + ch]);
    }
    auto draw_pairs = [&](int n0) {
        const int n = n0 + lane;
        if (n < total) {
            int j, k;
            pair_jk(p.seed, (uint32_t)gr.sample, (uint32_t)(base + n / half), (uint32_t)(n % half), N, j, k);
            pairs[n & 63] = j | (k << 16);
        }
        __syncwarp();
    };
    auto draw_proposals = [&](int n0) {  // lane = (chain, update n0 + lane / GC)
        const int n = n0 + wq;
        if (n < total) draws[(n % (2 * UB)) * GC + c] = draw_proposal<float>(p.seed, cid, (uint32_t)(base + n / half), (uint32_t)(n % half));
        __syncwarp();
    };
    // update n's lists into buffer b (one lane); sizes are multiples of 16 bytes
    auto copy_lists = [&](int n, int b) {
        const int jk = pairs[n & 63], j = jk & 0xffff, k = jk >> 16, pi = tri_index(j, k, N);
        const int x0 = __ldg(xoff + pi), nx = __ldg(xoff + pi + 1) - x0;
        const uint32_t bj = (uint32_t)(choff[j + 1] - choff[j]) * 32u, bk = (uint32_t)(choff[k + 1] - choff[k]) * 32u, bx = (uint32_t)nx * 16u;
        s_nx[b] = nx;
        unsigned char *dst = smem + lay.list + b * lay.list_bytes;
        mbar_arrive_expect_tx(&lbar[b], bj + bk + bx);
        if (bj) bulk_g2s(dst, chunks + 2 * choff[j], bj, &lbar[b]);
        if (bk) bulk_g2s(dst + bj, chunks + 2 * choff[k], bk, &lbar[b]);
        if (bx) bulk_g2s(smem + lay.cross + b * lay.cross_bytes, cross + x0, bx, &lbar[b]);
    };
    // proposal of update n after update n - 1 (proposals Q) was rejected (v = 0) or accepted (v = 1), lane = (chain, v)
    auto propose = [&](int n, int jkq, unsigned mask, bool first) {
        const int v = wq;
        if (v < 2 && c < gr.count) {
            const int jk = pairs[n & 63], j = jk & 0xffff, k = jk >> 16;
            float2 aj = amp[j * GC + c], ak = amp[k * GC + c];
            if (!first && v) {
                const WarpProposal &Q = prop[((n & 1) ^ 1) * 2 * GC + ((mask >> c) & 1u) * GC + c];
                const int jq = jkq & 0xffff, kq = jkq >> 16;
                if (j == jq) aj = Q.nj; else if (j == kq) aj = Q.nk;
                if (k == jq) ak = Q.nj; else if (k == kq) ak = Q.nk;
            }
            const Proposal<float> P = finish_proposal<float>(draws[(n % (2 * UB)) * GC + c], aj, ak);
            WarpProposal &o = prop[(n & 1) * 2 * GC + v * GC + c];
            o.aj = aj; o.ak = ak; o.nj = P.nj; o.nk = P.nk; o.U = P.U;
        }
        __syncwarp();
    };
    if (helper && total > 0) {
        draw_pairs(0);
        draw_proposals(0);
        propose(0, 0, 0u, true);
        if (lane == 0) copy_lists(0, 0);
    }
    __syncthreads();
    unsigned mask = 0u;  // chains that accepted the previous update
    int sw = 0, u = 0;
    for (int n = 0; n < total; ++n) {
        const int jk = pairs[n & 63], j = jk & 0xffff, k = jk >> 16;
        const int b = nbuf == 2 ? (n & 1) : 0;
        const WarpProposal &P = prop[(n & 1) * 2 * GC + ((mask >> c) & 1u) * GC + c];
        const bool traced = tr_at == base + sw + 1 && u == tr_u;
        if (helper) {
            if ((n & 31) == 0) draw_pairs(n + 32);
            if (n + 1 < total) {
                if (nbuf == 2 && lane == 0) copy_lists(n + 1, b ^ 1);
                if ((n + 1) % UB == 0) draw_proposals(n + 1);
                propose(n + 1, jk, mask, false);
            }
        } else {
            const float2 dj = make_float2(P.nj.x - P.aj.x, P.nj.y - P.aj.y), dk = make_float2(P.nk.x - P.ak.x, P.nk.y - P.ak.y);
            float2 hj = make_float2(0.f, 0.f), hk = make_float2(0.f, 0.f);
            float cr = 0.f;
            const bool landed = mbar_wait_bounded(&lbar[b], (uint32_t)(nbuf == 2 ? (n >> 1) & 1 : n & 1), p.ctl, 33, abort_flag);
            if (landed) {
                const int4 *L = reinterpret_cast<const int4 *>(smem + lay.list + b * lay.list_bytes);
                const int ncj = choff[j + 1] - choff[j], nc = ncj + choff[k + 1] - choff[k];
                auto chunk = [&](int i, float2 &h) {
                    const int4 q = L[2 * i];
                    const float4 Jv = *reinterpret_cast<const float4 *>(L + 2 * i + 1);
                    const float2 g0 = pp[(q.x & 0xffff) * GC + c], g1 = pp[((unsigned)q.x >> 16) * GC + c];
                    const float2 g2 = pp[(q.y & 0xffff) * GC + c], g3 = pp[((unsigned)q.y >> 16) * GC + c];
                    const float2 m = amp[q.z * GC + c];
                    const float ax = fmaf(Jv.w, g3.x, fmaf(Jv.z, g2.x, fmaf(Jv.y, g1.x, Jv.x * g0.x)));
                    const float ay = fmaf(Jv.w, g3.y, fmaf(Jv.z, g2.y, fmaf(Jv.y, g1.y, Jv.x * g0.y)));
                    h.x = fmaf(m.x, ax, fmaf(m.y, ay, h.x));
                    h.y = fmaf(m.x, ay, fmaf(-m.y, ax, h.y));
                };
                int i = worker;
                for (; i < ncj; i += NWK) chunk(i, hj);
                for (; i < nc; i += NWK) chunk(i, hk);
                // quadruplets holding both modes: Re(J dx_lo dx_hi f_x f_y), conjugated by the flag bits 0..3
                const int4 *X = reinterpret_cast<const int4 *>(smem + lay.cross + b * lay.cross_bytes);
                const int nx = s_nx[b];
                const float2 dlo = j < k ? dj : dk, dhi = j < k ? dk : dj;
                for (int e = worker; e < nx; e += NWK) {
                    const int4 q = X[e];
                    float2 fx = amp[q.x * GC + c], fy = amp[q.y * GC + c], l = dlo, h = dhi;
                    if (q.z & 1) l.y = -l.y;
                    if (q.z & 2) h.y = -h.y;
                    if (q.z & 4) fx.y = -fx.y;
                    if (q.z & 8) fy.y = -fy.y;
                    const float2 d2 = cmulf(l, h), f2_ = cmulf(fx, fy);
                    cr += __int_as_float(q.w) * (d2.x * f2_.x - d2.y * f2_.y);
                }
            }
            float v = dj.x * hj.x + dj.y * hj.y + dk.x * hk.x + dk.y * hk.y + cr;
#pragma unroll
            for (int o = GC; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (wq == 0) part[((n & 1) * FW + warp) * GC + c] = v;
            if (traced) {  // the record's sums, added over the warps in FP64, and the state before the update
                const float t5[5] = {hj.x, hj.y, hk.x, hk.y, cr};
#pragma unroll
                for (int e = 0; e < 5; ++e) {
                    float s = t5[e];
                    for (int o = GC; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (wq == 0 && c < gr.count) atomicAdd(p.trace + (int64_t)cid * kTraceRec + 2 + e, (double)s);
                }
                for (int ch = 0; ch < gr.count; ++ch) {
                    const uint32_t id = __shfl_sync(0xffffffffu, cid, ch);
                    double2 *st = reinterpret_cast<double2 *>(p.trace + (int64_t)p.n_chains * kTraceRec) + sd.a_off +
                                  (int64_t)(id - (uint32_t)sd.chain0) * N;
                    for (int x = tid; x < N; x += FW * 32) st[x] = make_double2((double)amp[x * GC + ch].x, (double)amp[x * GC + ch].y);
                }
            }
        }
        __syncthreads();
        // decision, in every warp alike
        float s = 0.f;
#pragma unroll
        for (int w0 = 0; w0 < FW; w0 += WPW)
            if (w0 + wq < FW) s += part[((n & 1) * FW + w0 + wq) * GC + c];
#pragma unroll
        for (int o = GC; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float dH = -cc * s;
        const bool acc = c < gr.count && metropolis_accept(dH, beta, P.U);
        if (traced && warp == 0 && wq == 0 && c < gr.count) {
            double *rec = p.trace + (int64_t)cid * kTraceRec;
            rec[0] = j; rec[1] = k;
            rec[10] = P.nj.x; rec[11] = P.nj.y; rec[12] = P.nk.x; rec[13] = P.nk.y;
            rec[14] = P.U; rec[15] = dH; rec[16] = acc ? 1.0 : 0.0; rec[17] = beta; rec[18] = E; rec[19] = 1.0;
        }
        if (acc) {
            for (int i = worker; i < 2 * N; i += (FW + 1) * WPW) {  // the helper's lanes too
                const bool fk = i >= N;
                const int m = fk ? i - N : i, l = fk ? k : j;
                if (m == l || (fk && m == j)) continue;
                const float2 nl = fk ? P.nk : P.nj, nm = (!fk && m == k) ? P.nk : amp[m * GC + c];
                pp[tri_index(l, m, N) * GC + c] = l < m ? tab_product(nl, nm) : tab_product(nm, nl);
            }
            if (warp == 0 && wq == 0) {
                amp[j * GC + c] = P.nj;
                amp[k * GC + c] = P.nk;
                E += (double)dH;
                ++n_acc;
            }
        }
        mask = __ballot_sync(0xffffffffu, acc && wq == 0);
        if (nbuf == 1 && helper && lane == 0 && n + 1 < total) copy_lists(n + 1, 0);
        __syncthreads();
        if (++u == half) {
            u = 0; ++sw;
            const long long done = base + sw;
            if (p.measure_every > 0 && done % p.measure_every == 0 && sw < p.n_sweeps) {
                const int kk = (int)(done / p.measure_every - base / p.measure_every - 1);
                if (kk >= 0 && kk < p.n_snap_max) {
                    float2 *dst = p.snap_a + (int64_t)kk * p.a_total + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
                    for (int i = tid; i < N * gr.count; i += NT) {
                        const int ch = i / N, x = i - ch * N;
                        dst[i] = amp[x * GC + ch];
                    }
                    if (tid < gr.count) p.snap_E[(int64_t)kk * p.n_chains + gr.chain0 + tid] = E;
                }
                __syncthreads();
            }
        }
    }
    // never leave bulk copies in flight behind an exiting block (only possible after a wait gave up)
    if (helper && lane == 0 && *abort_flag)
        for (int n = max(0, total - nbuf); n < total; ++n) {
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(&lbar[nbuf == 2 ? n & 1 : 0], (uint32_t)(nbuf == 2 ? (n >> 1) & 1 : n & 1)) && global_ns() - t0 < kWaitNs) {
            }
        }
    for (int i = tid; i < N * gr.count; i += NT) {
        const int ch = i / N, x = i - ch * N;
        A[i] = amp[x * GC + ch];
    }
    if (tid < gr.count) {
        const int slot = gr.chain0 + tid;
        if (!isfinite(E)) record_error(p.ctl, kErrNaN, 30);
        p.E[slot] = E;
        p.mc_acc[slot] += n_acc;
        p.mc_att[slot] += (unsigned long long)total;
    }
}

// Full energies of the chains of a group (optionally after rescaling to sum |a|^4 = N): each lane sums
// J_q Re(conj(a_q0) a_q1 a_q2 conj(a_q3)) for its chain over a share of the quadruplets, products in FP32,
// couplings and sums in FP64.
__global__ void __launch_bounds__(kGThreads) graph_energy_kernel(GraphParams p) {
    extern __shared__ float2 ga[];
    __shared__ double redd[kGWarps][kGG];
    __shared__ double s_f[kGG];
    const GroupDev gr = p.groups[blockIdx.x];
    const SampleDev sd = p.samples[gr.sample];
    const int N = sd.N, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int c = lane % kGG, worker = warp * (32 / kGG) + lane / kGG;
    float2 *A = p.a + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
    for (int i = tid; i < N * kGG; i += kGThreads) {
        const int x = i / kGG, cc = i % kGG;
        ga[x * kGRS + cc] = cc < gr.count ? A[(int64_t)cc * N + x] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (p.renorm) {
        double s4 = 0.0;
        for (int x = worker; x < N; x += kGWorkers) {
            const float2 v = ga[x * kGRS + c];
            const double uu = (double)v.x * v.x + (double)v.y * v.y;
            s4 += uu * uu;
        }
        for (int o = kGG; o < 32; o <<= 1) s4 += __shfl_xor_sync(0xffffffffu, s4, o);
        if (lane < kGG) redd[warp][c] = s4;
        __syncthreads();
        if (tid < kGG) {
            double t = 0.0;
            for (int w = 0; w < kGWarps; ++w) t += redd[w][tid];
            if (tid < gr.count && (!(t > 0.0) || !isfinite(t))) record_error(p.ctl, kErrNaN, 31);
            s_f[tid] = tid < gr.count ? sqrt(sqrt((double)N / t)) : 1.0;
        }
        __syncthreads();
        for (int i = tid; i < N * gr.count; i += kGThreads) {
            const int cc = i / N, x = i % N;
            const double f = s_f[cc];
            float2 v = ga[x * kGRS + cc];
            v = make_float2((float)((double)v.x * f), (float)((double)v.y * f));
            ga[x * kGRS + cc] = v;
            A[(int64_t)cc * N + x] = v;
        }
        __syncthreads();
    }
    const int4 *quads = p.quads + sd.q_off;
    const double *Jd = p.Jd + sd.q_off;
    double acc = 0.0;
    for (int64_t q = worker; q < sd.nq; q += kGWorkers) {
        const int4 Q = __ldg(quads + q);
        const float2 t = cmulf(cmulf(fac(ga[Q.x * kGRS + c], 0), ga[Q.y * kGRS + c]),
                               cmulf(ga[Q.z * kGRS + c], fac(ga[Q.w * kGRS + c], 3)));
        acc += __ldg(Jd + q) * (double)t.x;
    }
    for (int o = kGG; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane < kGG) redd[warp][c] = acc;
    __syncthreads();
    if (tid < gr.count) {
        double t = 0.0;
        for (int w = 0; w < kGWarps; ++w) t += redd[w][tid];
        const double Ec = -p.cc * t;
        const int slot = gr.chain0 + tid;
        if (!isfinite(Ec)) record_error(p.ctl, kErrNaN, 32);
        if (p.E_state) p.E_state[slot] = Ec;
        if (p.E_out) p.E_out[slot] = Ec;
    }
}

namespace {
// Records of an update (twice the largest degree) up to which a chain gets a block of its own (graph_warp_kernel): against the
// pair table with 8 chains per block, and against what remains where that table does not fit.  GB300, us per sweep, own
// block / other kernel.  Table: sparse N = 48, 1024 and 4096 chains, 120 records 27 / 40 and 75 / 143, 186 39 / 42 and
// 112 / 150, 268 50 / 42 and 144 / 151, 352 67 / 43 and 192 / 157.  Table of 4 chains, N = 96: 190 76 / 129 and 217 / 439,
// 314 113 / 138 and 331 / 470.  Group kernel, N = 256: 80 91 / 292 and 275 / 1143, 272 241 / 314 and 724 / 1237, 418
// 380 / 347 and 1145 / 1364.  Against the 8-chain table the line would lie near 200 records at 1024 chains and near 290 at 4096;
// 256 for both gives up to 20% at one and 5% at the other.
constexpr int kWarpMaxRec = 256, kWarpMaxAlone = 352;
constexpr size_t kGraphSmemMax = 227 * 1024 - 8 * 1024;  // dynamic part (the static reduction table aside)

// Whether the pair-table kernel's lists are worth building (their sizes then decide): the products of 4 chains and the two
// lists of an update (32 bytes per four records) fit.
}  // namespace
bool graph_table_candidate(int maxN, int max_deg) {
    const size_t pairs = (size_t)maxN * (maxN - 1) / 2 * sizeof(float2), lists = (size_t)2 * max_deg * 8;
    return 2 * max_deg > (8 * pairs + lists < kGraphSmemMax ? kWarpMaxRec : kWarpMaxAlone) && 4 * pairs + lists < kGraphSmemMax;
}
namespace {
// Shape of the pair-table kernel: chains per block, list buffers (two when they fit, so that an update's lists arrive
// during the one before).  8 chains per block read each record once for all 8; 4 where the products of 8 do not fit.
// 512 threads: every warp repeats the decision, so more warps cost more than they hide (N = 64, 1024 chains: 1024
// threads 142 us per sweep, 768 117, 512 108.7, 384 105.6, 256 113; two blocks of 4 chains per SM 121).
constexpr int kTabThreads = 512, kTabFW = kTabThreads / 32 - 1;
struct TabShape {
    int GC, nbuf;
    size_t smem;
};
bool table_shape(const GraphParams &p, TabShape *out) {
    for (int GC : {8, 4})
        for (int nbuf : {2, 1}) {
            const size_t sm = tab_smem(GC, kTabFW, p.maxN, p.max_chunks, p.max_cross, nbuf).total;
            if (sm <= kGraphSmemMax) {
                *out = TabShape{GC, nbuf, sm};
                return true;
            }
        }
    return false;
}
int graph_variant(const GraphParams &p) {
    TabShape t;
    const bool table = p.chunks && table_shape(p, &t);
    if (2 * p.max_deg <= (table && t.GC == 8 ? kWarpMaxRec : kWarpMaxAlone)) return kWarp;
    if (table) return kTable;
    if (graph_smem(p.maxN, 2 * p.max_deg).total <= kGraphSmemMax) return kStage;
    return kPlain;
}
size_t variant_smem(int var, const GraphParams &p) {
    TabShape t;
    if (var == kWarp) return (size_t)p.maxN * sizeof(float2);
    if (var == kTable && table_shape(p, &t)) return t.smem;
    return graph_smem(p.maxN, var == kStage ? 2 * p.max_deg : 0).total;
}
}  // namespace

// The limits are the kernels' largest, not this context's: they belong to the kernel, and contexts of other sizes launch it too.
cudaError_t graph_prepare(const GraphParams &p) {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const int most = (int)kGraphSmemMax, mode = 2048 * (int)sizeof(float2);
    cudaError_t e = cudaSuccess;
    TabShape t;
    switch (graph_variant(p)) {
        case kWarp: e = cudaFuncSetAttribute(graph_warp_kernel, at, mode); break;
        case kTable:
            table_shape(p, &t);
            e = t.GC == 8 ? cudaFuncSetAttribute(graph_table_kernel<8, kTabThreads>, at, most)
                          : cudaFuncSetAttribute(graph_table_kernel<4, kTabThreads>, at, most);
            break;
        case kStage: e = cudaFuncSetAttribute(graph_sweep_kernel<kStage>, at, most); break;
        default: e = cudaFuncSetAttribute(graph_sweep_kernel<kPlain>, at, most);
    }
    if (e == cudaSuccess) e = cudaFuncSetAttribute(graph_energy_kernel, at, kGRS * mode);
    return e;
}

cudaError_t launch_graph_sweep(const GraphParams &p0, int n_groups, cudaStream_t s) {
    if (n_groups <= 0) return cudaSuccess;
    GraphParams p = p0;
    const int var = graph_variant(p);
    const size_t sm = variant_smem(var, p);
    if (var == kWarp) graph_warp_kernel<<<p.n_chains, 64, sm, s>>>(p);
    else if (var == kTable) {
        TabShape t;
        table_shape(p, &t);
        p.tab_nbuf = t.nbuf;
        if (t.GC == 8) graph_table_kernel<8, kTabThreads><<<n_groups, kTabThreads, sm, s>>>(p);
        else graph_table_kernel<4, kTabThreads><<<2 * n_groups, kTabThreads, sm, s>>>(p);
    } else if (var == kStage) graph_sweep_kernel<kStage><<<n_groups, kGThreads, sm, s>>>(p);
    else graph_sweep_kernel<kPlain><<<n_groups, kGThreads, sm, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_graph_energy(const GraphParams &p, int n_groups, cudaStream_t s) {
    if (n_groups <= 0) return cudaSuccess;
    const size_t sm = (size_t)p.maxN * kGRS * sizeof(float2);
    graph_energy_kernel<<<n_groups, kGThreads, sm, s>>>(p);
    return cudaGetLastError();
}

}  // namespace ptgb
