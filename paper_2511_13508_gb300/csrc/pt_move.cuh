// pt_move.cuh -- complex arithmetic, the pair proposal and the Metropolis test, shared by the sweep kernels of
// the comb graph (arXiv 2511.13508, Sec. III.A.1).
#pragma once
#include "pt_common.cuh"

namespace ptgb {

// ------------------------------------------------------------------------------------------------
// complex arithmetic on float2/double2
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
    V r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
template <typename V> __device__ __forceinline__ V cmulc(V a, V b) {  // conj(a) * b
    V r;
    r.x = a.x * b.x + a.y * b.y;
    r.y = a.x * b.y - a.y * b.x;
    return r;
}
template <typename V, typename T> __device__ __forceinline__ void caxpy(V &acc, T s, V z) {
    acc.x = fma(s, z.x, acc.x);
    acc.y = fma(s, z.y, acc.y);
}
template <typename V> __device__ __forceinline__ void cadd(V &acc, V z) { acc.x += z.x; acc.y += z.y; }

// ------------------------------------------------------------------------------------------------
// Proposal of a pair move and Metropolis test (Sec. III.A.1, readings R3 and R6).
template <typename real> struct Proposal {
    typename vec2<real>::type aj, ak, nj, nk;  // old and proposed amplitudes
    real U;
};

// The pair move of Sec. III.A.1 in two parts: draw_proposal takes the random numbers of (chain, sweep, update)
// -- the angles as sqrt(cos theta), sqrt(sin theta), the phases as (cos, sin), and the Metropolis uniform U -- and
// needs no state, so the copy warp draws it ahead of the update; finish_proposal scales it by
// K = (|a_j|^4 + |a_k|^4)^(1/4) of the chain's current amplitudes (mode j receives K sqrt(cos theta)).
template <typename real> struct ProposalDraw {
    real sqc, sqs, cj, sj, ck, sk, U, pad;
};

template <typename real>
__device__ __forceinline__ ProposalDraw<real> draw_proposal(uint64_t seed, uint32_t chain_id, uint32_t sweep,
                                                            uint32_t update);

template <>
__device__ __forceinline__ ProposalDraw<float> draw_proposal<float>(uint64_t seed, uint32_t chain_id, uint32_t sweep,
                                                                    uint32_t update) {
    ProposalDraw<float> D;
    const u32x4 w = draw(seed, chain_id, sweep, update, kTagPropose);
    const float kInv = 2.3283064365386963e-10f;
    const float fj = ((float)w.x + 0.5f) * kInv, fk = ((float)w.y + 0.5f) * kInv, ft = ((float)w.z + 0.5f) * kInv;
    float st, ct;
    sincospif(2.0f * fj, &D.sj, &D.cj);
    sincospif(2.0f * fk, &D.sk, &D.ck);
    sincospif(0.5f * ft, &st, &ct);
    D.sqc = sqrtf(ct);
    D.sqs = sqrtf(st);
    D.U = ((float)w.w + 0.5f) * kInv;
    D.pad = 0.f;
    return D;
}

template <>
__device__ __forceinline__ ProposalDraw<double> draw_proposal<double>(uint64_t seed, uint32_t chain_id,
                                                                      uint32_t sweep, uint32_t update) {
    ProposalDraw<double> D;
    const u32x4 w = draw(seed, chain_id, sweep, update, kTagPropose);
    const double phj = kTwoPi * u01(w.x), phk = kTwoPi * u01(w.y), th = kHalfPi * u01(w.z);
    D.sqc = sqrt(cos(th));
    D.sqs = sqrt(sin(th));
    sincos(phj, &D.sj, &D.cj);
    sincos(phk, &D.sk, &D.ck);
    D.U = u01(w.w);
    D.pad = 0.0;
    return D;
}

template <typename real>
__device__ __forceinline__ Proposal<real> finish_proposal(const ProposalDraw<real> &D, typename vec2<real>::type aj,
                                                          typename vec2<real>::type ak) {
    Proposal<real> P;
    P.aj = aj; P.ak = ak;
    // fused multiply-adds written out, so that every kernel rounds a proposal alike
    const real uj = fma(aj.x, aj.x, aj.y * aj.y), uk = fma(ak.x, ak.x, ak.y * ak.y);
    real K;
    if constexpr (sizeof(real) == 4) K = sqrtf(sqrtf(fma(uj, uj, uk * uk)));
    else K = sqrt(sqrt(fma(uj, uj, uk * uk)));
    const real Aj = K * D.sqc, Ak = K * D.sqs;
    P.nj.x = Aj * D.cj; P.nj.y = Aj * D.sj;
    P.nk.x = Ak * D.ck; P.nk.y = Ak * D.sk;
    P.U = D.U;
    return P;
}

__device__ __forceinline__ bool metropolis_accept(float dH, float beta, float U) {
    return dH <= 0.0f || U < expf(-beta * dH);
}
__device__ __forceinline__ bool metropolis_accept(double dH, double beta, double U) {
    return dH <= 0.0 || U < exp(-beta * dH);
}

}  // namespace ptgb
