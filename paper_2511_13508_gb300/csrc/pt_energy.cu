// pt_energy.cu -- full energies of FP32 chains on the comb graph (the resync of a run; arXiv 2511.13508, Eq. (4)).
//
// Every quadruplet once, at its smallest mode l:  H = -cc sum_l Re( conj(a_l) sum_m conj(a_m) acc_l[l+m] ),
// acc_l[s] = sum over the pairs {x, s-x}, x > l, of J_l[s][x] a_x a_{s-x}.  A pair product belongs to the sum s alone, not
// to l: a warp forms the products of one 8x8 tile (8 sums, 8 columns) of its chains once, keeps them in registers, and runs
// over the modes l that use the tile; a coupling term is then two multiply-adds (paired FP32, two sums at once) instead of
// six.  The coupling blocks of (tile, l) come through a ring of asynchronous copies per warp, kept deep: with direct
// loads the kernel waited on L2.  Products and row sums in FP32, the sums over tiles and modes in FP64.
// GB300, N = 256, 8 samples x 96 chains, the whole call: 902 us with a block per (mode, tile) and direct loads, 452 now.
#include <cstdint>
#include "pt_common.cuh"
#include "pt_kernels.h"

namespace ptgb {

namespace {

constexpr int kJS = JStride<float>::value;
constexpr int kEWarps = 8;

template <int G> __host__ __device__ constexpr int erow_stride() { return G == 8 ? G + 1 : G; }

struct EnergySmem {
    size_t win, amp, red, ring, total;
};
template <int G> __host__ __device__ EnergySmem energy_smem(int maxN, int depth) {
    EnergySmem m;
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o += (b + 127) / 128 * 128; return at; };
    m.win = take((size_t)(maxN + 2 * APAD) * G * sizeof(float4));
    m.amp = take((size_t)(maxN + 2 * APAD) * erow_stride<G>() * sizeof(float2));
    m.red = take((size_t)kEWarps * G * sizeof(double));
    m.ring = take((size_t)kEWarps * depth * (32 / G) * kJS * sizeof(float));
    m.total = o;
    return m;
}

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

template <int kDepth> __device__ __forceinline__ void wait_oldest() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
}

}  // namespace

// A block is part `blockIdx.x % parts` of a group; its warps take the items (tile, run of kEnergySeg modes) in turn.  Lane:
// chain c = lane % G, worker lane / G; the workers of a warp share the tile and take every (32/G)-th mode of the run.
template <int G, int kDepth>
__global__ void __launch_bounds__(kEWarps * 32, 1) energy_tile_kernel(EnergyParams p) {
    constexpr int RS = erow_stride<G>(), WPW = 32 / G;
    extern __shared__ __align__(128) unsigned char smem[];
    const EnergySmem lay = energy_smem<G>(p.maxN, kDepth);
    float4 *win = reinterpret_cast<float4 *>(smem + lay.win);
    float2 *amp = reinterpret_cast<float2 *>(smem + lay.amp);
    double *red = reinterpret_cast<double *>(smem + lay.red);
    const int part = (int)(blockIdx.x % (unsigned)p.parts), group = (int)(blockIdx.x / (unsigned)p.parts);
    const GroupDev gr = p.groups[group];
    const SampleDev sd = p.samples[gr.sample];
    const int N = sd.N, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c = lane % G, wq = lane / G;
    float *ring = reinterpret_cast<float *>(smem + lay.ring) + (size_t)warp * kDepth * WPW * kJS;
    const float2 *A = reinterpret_cast<const float2 *>(p.a) + sd.a_off + (int64_t)(gr.chain0 - sd.chain0) * N;
    const int rows = N + 2 * APAD;
    for (int i = tid; i < rows * G; i += kEWarps * 32) {
        const int ch = i / rows, R = i - ch * rows, x = R - APAD;
        amp[R * RS + ch] = (x >= 0 && x < N && ch < gr.count) ? A[(int64_t)ch * N + x] : f2(0.f, 0.f);
    }
    __syncthreads();
    for (int i = tid; i < rows * G; i += kEWarps * 32) {
        const int R = i / G, ch = i % G;
        const float2 a = amp[R * RS + ch], b = R + 1 < rows ? amp[(R + 1) * RS + ch] : f2(0.f, 0.f);
        win[i] = make_float4(a.x, b.x, a.y, b.y);
    }
    __syncthreads();
    const float *J = reinterpret_cast<const float *>(p.J);
    const int *bo = p.bo + sd.tab_off, *mode_blk = p.mode_blk + sd.mode_off, *seg = p.eseg + sd.seg_off;
    const uint32_t *binfo = p.blkinfo + sd.blk_off;
    const int items = seg[sd.nblk], nw = kEWarps * p.parts;
    double e = 0.0;
    int b = 0;
    for (int it = part * kEWarps + warp; it < items; it += nw) {
        while (seg[b + 1] <= it) ++b;
        const uint32_t info = binfo[b];
        const int st = (int)(info >> 16), s0 = st * TS, x0 = (int)(info & 0xffffu) * TX;
        // modes that use the tile: l < x for some column, and the tile lies in l's run
        const int l_lo = max(0, s0 - N + 1) + (it - seg[b]) * kEnergySeg, l_hi = min(min(x0 + TX - 1, N), l_lo + kEnergySeg);
        const int steps = (l_hi - l_lo + WPW - 1) / WPW;
        // the block of mode l: J_l's run starts at the blocks of s-tile l / 8
        auto copy = [&](int i) {
            const int l = l_lo + i * WPW + wq;
            if (i < steps && l < l_hi) {
                const float *src = J + (sd.J_off + mode_blk[l] + b - bo[l / TS]) * kJS;
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + ((i % kDepth) * WPW + wq) * kJS);
#pragma unroll
                for (int k = 0; k < (16 + G - 1) / G; ++k) {
                    const int at = (c + k * G) * 4;
                    if (G <= 16 || c < 16)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + at * 4), "l"(src + at) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int i = 0; i < kDepth - 1; ++i) copy(i);
        // products of the tile, columns 2h + pi with the window at y = s0 - x0 - i + 2q
        float2 zx[TX][TS / 2], zy[TX][TS / 2];
        const int ybase = s0 - x0 + APAD;
#pragma unroll
        for (int i = 0; i < TX; ++i) {
            const float2 ax = amp[(x0 + i + APAD) * RS + c];
            const float2 sx = f2(ax.x, ax.x), sy = f2(ax.y, ax.y), ny = f2(-ax.y, -ax.y);
#pragma unroll
            for (int q = 0; q < TS / 2; ++q) {
                const float4 w = win[(ybase + 2 * q - i) * G + c];
                const float2 wx = f2(w.x, w.y), wy = f2(w.z, w.w);
                zx[i][q] = __ffma2_rn(sx, wx, __fmul2_rn(ny, wy));
                zy[i][q] = __ffma2_rn(sx, wy, __fmul2_rn(sy, wx));
            }
        }
        for (int i = 0; i < steps; ++i) {
            copy(i + kDepth - 1);
            wait_oldest<kDepth>();
            __syncwarp();
            const int l = l_lo + i * WPW + wq;
            if (l < l_hi) {
                const float *Jl = ring + ((i % kDepth) * WPW + wq) * kJS;
                float2 ax[TS / 2], ay[TS / 2];
#pragma unroll
                for (int q = 0; q < TS / 2; ++q) ax[q] = ay[q] = f2(0.f, 0.f);
                const int skip = l - x0;  // columns up to here are pairs whose smaller mode is <= l: counted at that mode
#pragma unroll
                for (int k = 0; k < TX; ++k) {
                    float4 u = *reinterpret_cast<const float4 *>(Jl + k * TS), v = *reinterpret_cast<const float4 *>(Jl + k * TS + 4);
                    if (k <= skip) u = v = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float2 j2[4] = {f2(u.x, u.y), f2(u.z, u.w), f2(v.x, v.y), f2(v.z, v.w)};
#pragma unroll
                    for (int q = 0; q < TS / 2; ++q) {
                        ax[q] = __ffma2_rn(j2[q], zx[k][q], ax[q]);
                        ay[q] = __ffma2_rn(j2[q], zy[k][q], ay[q]);
                    }
                }
                // sum_m conj(a_m) acc over the 8 sums (couplings are zero where m = s - l is no partner), then Re(conj(a_l) .)
                float2 tx = f2(0.f, 0.f), ty = f2(0.f, 0.f), tn = f2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < TS / 2; ++q) {
                    const float4 w = win[(s0 + 2 * q - l + APAD) * G + c];
                    const float2 mx = f2(w.x, w.y), my = f2(w.z, w.w);
                    tx = __ffma2_rn(mx, ax[q], tx);
                    tx = __ffma2_rn(my, ay[q], tx);
                    ty = __ffma2_rn(mx, ay[q], ty);
                    tn = __ffma2_rn(my, ax[q], tn);
                }
                const float2 al = amp[(l + APAD) * RS + c];
                e += (double)(al.x * (tx.x + tx.y) + al.y * ((ty.x + ty.y) - (tn.x + tn.y)));
            }
            __syncwarp();
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int o = G; o < 32; o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane < G) red[warp * G + c] = e;
    __syncthreads();
    if (tid < gr.count) {
        double t = 0.0;
        for (int w = 0; w < kEWarps; ++w) t += red[w * G + tid];
        p.part[((size_t)group * p.parts + part) * 32 + tid] = t;
    }
}

namespace {
template <int G, int kDepth> bool launch_depth(const EnergyParams &p, int ngroups, size_t limit, cudaStream_t s, cudaError_t *e) {
    const size_t sm = energy_smem<G>(p.maxN, kDepth).total;
    if (sm > limit) return false;
    *e = cudaFuncSetAttribute(energy_tile_kernel<G, kDepth>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
    if (*e != cudaSuccess) return true;
    energy_tile_kernel<G, kDepth><<<ngroups * p.parts, kEWarps * 32, sm, s>>>(p);
    *e = cudaGetLastError();
    return true;
}
template <int G> cudaError_t launch_g(const EnergyParams &p, int ngroups, cudaStream_t s) {
    int dev = 0, limit = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (launch_depth<G, 8>(p, ngroups, (size_t)limit, s, &e) || launch_depth<G, 2>(p, ngroups, (size_t)limit, s, &e)) return e;
    return cudaErrorInvalidConfiguration;
}
}  // namespace

cudaError_t launch_energy_tiles(int G, const EnergyParams &p, int ngroups, cudaStream_t s) {
    if (G == 8) return launch_g<8>(p, ngroups, s);
    if (G == 16) return launch_g<16>(p, ngroups, s);
    if (G == 32) return launch_g<32>(p, ngroups, s);
    return cudaErrorInvalidValue;
}

}  // namespace ptgb
