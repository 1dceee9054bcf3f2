// Hidden RMSNorm, fused residual + RMSNorm and SwiGLU: the element-wise operators around the
// attention and FFN blocks that the paper's operator table lists as unified operators.  All
// three touch every byte once and are bound by HBM traffic: 16-byte coalesced accesses, the
// whole row of a norm requested before anything is computed, and small CTAs so that enough of
// them are resident to keep the memory system busy.  A row's result depends on that row, the
// weight and eps only (fixed 128-thread reduction shape), never on the number of rows.
#include <cuda_bf16.h>

#include "tik_core.cuh"
#include "tik_internal.h"
#include "tik_ptx.cuh"

namespace tik {

constexpr int HN_THREADS = 128;
constexpr unsigned SW_VEC_MAX = 0xfffff000u;      // SwiGLU output vectors per launch

__device__ __forceinline__ void unpack8(const uint4& v, float* f) {
    const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(r[i] << 16);              // bf16 -> fp32 is exact
        f[2 * i + 1] = __uint_as_float(r[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack8(const float* f) {
    return make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]),
                      pack_bf16x2(f[6], f[7]));
}

// One CTA per row; NV = 16-byte vectors per thread (H <= 1024 * NV).
template <int NV, bool RESIDUAL>
__global__ void __launch_bounds__(HN_THREADS) rmsnorm_kernel(const NormParams p) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long row = blockIdx.x;
    const int nvec = p.H / 8;
    const uint4* x = reinterpret_cast<const uint4*>(p.x) + row * nvec;
    uint4* res = RESIDUAL ? reinterpret_cast<uint4*>(p.residual) + row * nvec : nullptr;
    const uint4* w = reinterpret_cast<const uint4*>(p.weight);
    uint4* y = reinterpret_cast<uint4*>(p.y) + row * nvec;
    __shared__ float warp_tot[4];
    pdl_wait();
    // Releases pass at one CTA per ~1.07 ns, so many rows that take less than that each go without (call after call: 9000 x
    // 512 6.2 us without and 10.1 with the release, 9000 x 2048 8.9 and 10.1; 9000 x 3584 21.4 and 20.3).
    if (gridDim.x <= 2048 || p.H * (RESIDUAL ? 2 : 1) >= 3072) pdl_launch_dependents();

    uint4 xv[NV], rv[RESIDUAL ? NV : 1];
#pragma unroll
    for (int j = 0; j < NV; ++j) {                           // the whole row is requested first
        const int v = tid + HN_THREADS * j;
        if (v < nvec) {
            xv[j] = x[v];
            if (RESIDUAL) rv[j] = res[v];
        }
    }
    float s[NV][8];
    float part = 0.0f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int v = tid + HN_THREADS * j;
        if (v < nvec) {
            unpack8(xv[j], s[j]);
            if (RESIDUAL) {
                float r[8];
                unpack8(rv[j], r);
#pragma unroll
                for (int e = 0; e < 8; ++e) s[j][e] = hn_residual_sum(s[j][e], r[e]);
                res[v] = pack8(s[j]);                        // exact: the sums are bf16 values
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) part = __fmaf_rn(s[j][e], s[j][e], part);
        }
    }
    part = hn_warp_total(part);
    if (lane == 0) warp_tot[warp] = part;
    __syncthreads();
    const float inv = prep_inv_rms(hn_block_total(warp_tot), 1.0f / static_cast<float>(p.H), p.eps);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int v = tid + HN_THREADS * j;
        if (v < nvec) {
            float wf[8], o[8];
            unpack8(w[v], wf);
#pragma unroll
            for (int e = 0; e < 8; ++e) o[e] = prep_norm(s[j][e], inv, wf[e]);
            y[v] = pack8(o);
        }
    }
}

// out[t][i] = silu(gu[t][i]) * gu[t][I + i]; 16-byte vectors of 8 outputs, SW_VPT per thread (a block
// covers 256 * SW_VPT consecutive vectors).  Large calls take four: all eight loads of a thread are
// issued before the arithmetic, 128 bytes per thread in flight (6.3 -> 6.9 TB/s on 32 768 x 27 648);
// small calls (decode) take one, which spreads them over more blocks.
// Inside an FFN the power limit holds the clock at 1.4 GHz and the kernel is bound by its instructions as much as by HBM,
// so outputs go two at a time (swiglu_value_x2), indices have 32 bits and a row is found by one division per thread.  One
// output at a time with a 64-bit division per vector -> this, us, alone out of HBM: 5999 x 18944 111.7 -> 106.0, 16000 x 8960
// 182 -> 139, 3001 x 27648 107 -> 84, 700 x 18944 22.6 -> 20.5.  The FFN around it: 5999 rows 2077 -> 2072 (within what runs of
// one side differ by), 16000 1308 -> 1290, 3000 x 8960 259.8 -> 255.0, 16 x 8960 24.5 -> 23.9; with the division and indices
// alone 2072, 1294, 257.3 and 24.3.
// Five blocks per SM: with four vectors the allocation is 48 registers then (nothing spilled), 56 otherwise, and four blocks
// have fewer bytes in flight (5999 x 18944 106 us both; 8000 x 12288 98, four blocks 102; 3001 x 27648 84, 87).
template <int SW_VPT>
__global__ void __launch_bounds__(256, 5) swiglu_kernel(const __nv_bfloat16* gu, __nv_bfloat16* out, unsigned nvec, unsigned vpr,
                                                        unsigned dt, unsigned dc) {
    const unsigned base = blockIdx.x * (256u * SW_VPT) + threadIdx.x;    // (nvec is at most SW_VEC_MAX: nothing wraps)
    pdl_wait();
    pdl_launch_dependents();
    // Row and column of a thread's first vector by one division, of the next ones, 256 = dt * vpr + dc vectors on, by
    // adding up: a 64-bit division per vector was a third of the instructions.
    unsigned t = base / vpr, c = base - t * vpr;
    uint4 gv[SW_VPT], uv[SW_VPT];
#pragma unroll
    for (int j = 0; j < SW_VPT; ++j) {
        if (base + 256 * j < nvec) {
            const uint4* row = reinterpret_cast<const uint4*>(gu) + 2ull * t * vpr;
            gv[j] = row[c];
            uv[j] = row[vpr + c];
        }
        t += dt;
        c += dc;
        if (c >= vpr) {
            c -= vpr;
            ++t;
        }
    }
#pragma unroll
    for (int j = 0; j < SW_VPT; ++j) {
        const unsigned idx = base + 256 * j;
        if (idx < nvec) {
            uint32_t w[4] = {gv[j].x, gv[j].y, gv[j].z, gv[j].w};
            const uint32_t uw[4] = {uv[j].x, uv[j].y, uv[j].z, uv[j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float o0, o1;
                swiglu_value_x2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u), __uint_as_float(uw[e] << 16),
                                __uint_as_float(uw[e] & 0xffff0000u), o0, o1);
                w[e] = pack_bf16x2(o0, o1);
            }
            reinterpret_cast<uint4*>(out)[idx] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

template <bool RESIDUAL>
static cudaError_t launch_rmsnorm_t(const NormParams& p, cudaStream_t stream) {
    const unsigned grid = static_cast<unsigned>(p.T);
    const int nv = (p.H / 8 + HN_THREADS - 1) / HN_THREADS;
    auto kern = nv <= 1 ? rmsnorm_kernel<1, RESIDUAL> : nv <= 2 ? rmsnorm_kernel<2, RESIDUAL>
              : nv <= 4 ? rmsnorm_kernel<4, RESIDUAL> : rmsnorm_kernel<8, RESIDUAL>;
    return launch_pdl(kern, dim3(grid), HN_THREADS, 0, stream, 1, p);
}

cudaError_t launch_rmsnorm(const NormParams& p, cudaStream_t stream) {
    if (p.T <= 0) return cudaSuccess;
    return p.residual ? launch_rmsnorm_t<true>(p, stream) : launch_rmsnorm_t<false>(p, stream);
}

cudaError_t launch_swiglu(const void* gu, void* out, long long T, int I, cudaStream_t stream) {
    const unsigned vpr = I / 8;                              // output vectors per row
    const auto* g = static_cast<const __nv_bfloat16*>(gu);
    auto* o = static_cast<__nv_bfloat16*>(out);
    // a launch takes as many rows as 32-bit vector indices count
    for (long long rows; T > 0; T -= rows, g += 2 * rows * I, o += rows * I) {
        rows = std::min<long long>(T, SW_VEC_MAX / vpr);
        const unsigned n = static_cast<unsigned>(rows * vpr);
        const bool large = n >= (1u << 20);
        cudaError_t e = launch_pdl(large ? swiglu_kernel<4> : swiglu_kernel<1>, dim3(large ? (n + 1023) / 1024 : (n + 255) / 256), 256, 0,
                                   stream, 1, g, o, n, vpr, 256 / vpr, 256 % vpr);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tik
