// Shared by the direct-difference kernels (fd_direct.cu: every column tile; fd_direct_listed.cu: tile lists).
#pragma once

#include "fd_internal.h"

namespace fd {

// Passes over the context's whole point set whose tile lists hold: kind 2 (by the boxes) or 4 (by what a degree pass noted).
fd_status apply_direct_listed(fd_ctx* c, const ApplyArgs& a, int kind);

namespace direct {

constexpr int kThr = 128;        // threads per CTA

template <class Kernel>
int resident(Kernel kernel, int smem, int most) {    // CTAs per SM, a property of the compiled kernel: asked once
    int n = 0;
    if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kThr, smem) != cudaSuccess || n < 1) n = 1;
    return n < most ? n : most;
}

inline int pick_bt(int bc) { return bc <= 4 ? 4 : bc <= 8 ? 8 : bc <= 16 ? 16 : bc <= 24 ? 24 : bc <= 32 ? 32 : bc <= 48 ? 48 : 64; }

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void copy16(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Kernel values of R rows and the point at sx[jj * DP4 ..].
template <int DP4, int R>
__device__ __forceinline__ void kernel_values(const float4* sx, int jj, const float4 (&xi)[R][DP4], float nbeta2, float (&kij)[R]) {
    float h[R];
#pragma unroll
    for (int r = 0; r < R; ++r) h[r] = 0.f;
#pragma unroll
    for (int k = 0; k < DP4; ++k) {
        const float4 xj = sx[jj * DP4 + k];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float d0 = xi[r][k].x - xj.x, d1 = xi[r][k].y - xj.y, d2 = xi[r][k].z - xj.z, d3 = xi[r][k].w - xj.w;
            h[r] = fmaf(d0, d0, h[r]); h[r] = fmaf(d1, d1, h[r]); h[r] = fmaf(d2, d2, h[r]); h[r] = fmaf(d3, d3, h[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) kij[r] = ex2_approx(h[r] * nbeta2);
}

// Sums of BT columns for R rows.  add(): sum[r][c] += kij[r] w[c].  64 columns use packed arithmetic (two columns an instruction: half the issue
// slots, the same time on the FMA pipe): N = 12000, D = 4: 744 -> 627 us a product, D = 32: 988 -> 930 (below 4500 points 2 to 4 % slower there).
// Narrower blocks are 2 to 8 % slower with it.
template <int R, int BT, bool PACKED = (BT > 48)>
struct Sums;
template <int R, int BT>
struct Sums<R, BT, false> {
    float v[R][BT];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < BT; ++c) v[r][c] = 0.f;
    }
    __device__ __forceinline__ void add(const float (&kij)[R], const float4* w) {
#pragma unroll
        for (int c4 = 0; c4 < BT / 4; ++c4) {
            const float4 w4 = w[c4];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r][4 * c4 + 0] = fmaf(kij[r], w4.x, v[r][4 * c4 + 0]);
                v[r][4 * c4 + 1] = fmaf(kij[r], w4.y, v[r][4 * c4 + 1]);
                v[r][4 * c4 + 2] = fmaf(kij[r], w4.z, v[r][4 * c4 + 2]);
                v[r][4 * c4 + 3] = fmaf(kij[r], w4.w, v[r][4 * c4 + 3]);
            }
        }
    }
    __device__ __forceinline__ float get(int r, int c) const { return v[r][c]; }
};
template <int R, int BT>
struct Sums<R, BT, true> {
    uint64_t v[R][BT / 2];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < BT / 2; ++c) v[r][c] = 0;
    }
    __device__ __forceinline__ void add(const float (&kij)[R], const float4* w) {
        uint64_t kk[R];
#pragma unroll
        for (int r = 0; r < R; ++r) kk[r] = pair2(kij[r], kij[r]);
#pragma unroll
        for (int c4 = 0; c4 < BT / 4; ++c4) {
            const ulonglong2 w4 = reinterpret_cast<const ulonglong2*>(w)[c4];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r][2 * c4] = fma2(kk[r], w4.x, v[r][2 * c4]);
#pragma unroll
            for (int r = 0; r < R; ++r) v[r][2 * c4 + 1] = fma2(kk[r], w4.y, v[r][2 * c4 + 1]);
        }
    }
    __device__ __forceinline__ float get(int r, int c) const {
        const float2 a = split2(v[r][c / 2]);
        return c & 1 ? a.y : a.x;
    }
};

}  // namespace direct

}  // namespace fd
