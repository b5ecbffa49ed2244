// fd_apply_general_static and its kernels: the split direct-difference block product with scratch of its own (see below).
// The ordinary direct-difference passes: fd_direct.cu.  This one keeps the earlier split (one row per thread, column ranges over
// gridDim.y, a second kernel adds the partials): its partials need no room beyond what the fixed array holds.
#include "fd_internal.h"

namespace fd {

namespace {

constexpr int kRows = 128;     // rows per CTA = threads per CTA
constexpr int kTJ = 64;        // points per column tile
constexpr int kFlushTiles = 32;  // column tiles between flushes of the fp32 tile accumulators

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// wp[j * BT + c] = right[j] * V[j + (c0 + c) * ldv] for c < bc, 0 for bc <= c < BT.
__global__ void k_pack_w(const float* __restrict__ V, int64_t ldv, const float* __restrict__ right, int64_t N,
                         int c0, int bc, int BT, float* __restrict__ wp) {
    __shared__ float tile[32][33];
    int64_t j0 = (int64_t)blockIdx.x * 32;
    int cb = blockIdx.y * 32;
    // read: threadIdx.x runs over j (coalesced along a column of V)
    for (int cc = threadIdx.y; cc < 32; cc += blockDim.y) {
        int c = cb + cc;
        int64_t j = j0 + threadIdx.x;
        float v = 0.0f;
        if (c < bc && j < N) {
            v = V[j + (int64_t)(c0 + c) * ldv];
            if (right) v *= right[j];
        }
        tile[cc][threadIdx.x] = v;
    }
    __syncthreads();
    // write: threadIdx.x runs over c (coalesced along a row of wp)
    for (int jj = threadIdx.y; jj < 32; jj += blockDim.y) {
        int c = cb + threadIdx.x;
        int64_t j = j0 + jj;
        if (c < BT && j < N) wp[j * BT + c] = tile[threadIdx.x][jj];
    }
}

// out[c * ld_out + i] = (left_i) * sum_j K_ij wp[j][c]   over this CTA's column range.
template <int DP4, int BT>
__global__ void __launch_bounds__(kRows)
k_simt(const float4* __restrict__ xrow, int64_t Nrow, const float4* __restrict__ xcol, int64_t N, float nbeta2,
       const float* __restrict__ wp, int64_t j_per_split, const float* __restrict__ left,
       float* __restrict__ out, int64_t ld_out, int64_t split_stride, int bstore) {
    __shared__ float4 sx[kTJ * DP4];
    __shared__ __align__(16) float sw[kTJ * BT];

    const int64_t i = (int64_t)blockIdx.x * kRows + threadIdx.x;
    const bool active = i < Nrow;
    float4 xi[DP4];
#pragma unroll
    for (int k = 0; k < DP4; ++k) xi[k] = active ? xrow[i * DP4 + k] : make_float4(0.f, 0.f, 0.f, 0.f);

    float acc[BT], acc_hi[BT];
#pragma unroll
    for (int c = 0; c < BT; ++c) { acc[c] = 0.f; acc_hi[c] = 0.f; }

    const int64_t jbeg = (int64_t)blockIdx.y * j_per_split;
    const int64_t jend = jbeg + j_per_split < N ? jbeg + j_per_split : N;
    int tiles_since_flush = 0;
    for (int64_t j0 = jbeg; j0 < jend; j0 += kTJ) {
        const int jn = (int)(jend - j0 < kTJ ? jend - j0 : kTJ);
        __syncthreads();
        for (int t = threadIdx.x; t < jn * DP4; t += kRows) sx[t] = xcol[j0 * DP4 + t];
        const float4* src = reinterpret_cast<const float4*>(wp + j0 * BT);
        float4* dst = reinterpret_cast<float4*>(sw);
        for (int t = threadIdx.x; t < jn * (BT / 4); t += kRows) dst[t] = src[t];
        __syncthreads();
#pragma unroll 2
        for (int jj = 0; jj < jn; ++jj) {
            float h = 0.f;
#pragma unroll
            for (int k = 0; k < DP4; ++k) {
                const float4 xj = sx[jj * DP4 + k];
                float d0 = xi[k].x - xj.x, d1 = xi[k].y - xj.y, d2 = xi[k].z - xj.z, d3 = xi[k].w - xj.w;
                h = fmaf(d0, d0, h); h = fmaf(d1, d1, h); h = fmaf(d2, d2, h); h = fmaf(d3, d3, h);
            }
            const float kij = ex2_approx(h * nbeta2);
#pragma unroll
            for (int c4 = 0; c4 < BT / 4; ++c4) {
                const float4 w = *reinterpret_cast<const float4*>(&sw[jj * BT + 4 * c4]);
                acc[4 * c4 + 0] = fmaf(kij, w.x, acc[4 * c4 + 0]);
                acc[4 * c4 + 1] = fmaf(kij, w.y, acc[4 * c4 + 1]);
                acc[4 * c4 + 2] = fmaf(kij, w.z, acc[4 * c4 + 2]);
                acc[4 * c4 + 3] = fmaf(kij, w.w, acc[4 * c4 + 3]);
            }
        }
        if (++tiles_since_flush == kFlushTiles) {
            // two-level summation keeps the rounding error of long column ranges at the 1e-7 level
#pragma unroll
            for (int c = 0; c < BT; ++c) { acc_hi[c] += acc[c]; acc[c] = 0.f; }
            tiles_since_flush = 0;
        }
    }
    if (!active) return;
    const float l = left ? left[i] : 1.0f;
    float* o = out + (int64_t)blockIdx.y * split_stride + i;
#pragma unroll
    for (int c = 0; c < BT; ++c)
        if (c < bstore) o[(int64_t)c * ld_out] = (acc_hi[c] + acc[c]) * l;
}

// Y[i + c * ldy] = left_i * sum_s part[s * split_stride + c * Nrow + i], s in a fixed order.
__global__ void k_reduce_block(const float* __restrict__ part, int splits, int64_t split_stride, int64_t Nrow, int bc,
                               const float* __restrict__ left, float* __restrict__ Y, int64_t ldy) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int c = blockIdx.y;
    if (i >= Nrow || c >= bc) return;
    float acc = 0.f;
    for (int s = 0; s < splits; ++s) acc += part[(int64_t)s * split_stride + (int64_t)c * Nrow + i];
    Y[i + (int64_t)c * ldy] = acc * (left ? left[i] : 1.0f);
}

struct SimtArgs {
    dim3 grid; cudaStream_t st;
    const float* x; int64_t N; float nbeta2; const float* wp; int64_t jps; const float* left; float* out;
    int64_t ld_out, split_stride; int bstore;
};

template <int DP4>
bool launch_simt_bt(int BT, const SimtArgs& a) {
    const float4* x = reinterpret_cast<const float4*>(a.x);
#define FD_CASE(B) case B: k_simt<DP4, B><<<a.grid, kRows, 0, a.st>>>(x, a.N, x, a.N, a.nbeta2, a.wp, a.jps, a.left, a.out, a.ld_out, a.split_stride, a.bstore); return true;
    switch (BT) {
        FD_CASE(4) FD_CASE(8) FD_CASE(16) FD_CASE(32)
        default: return false;
    }
#undef FD_CASE
}

bool launch_simt_any(int DP4, int BT, const SimtArgs& a) {
#define FD_CASE(Dq) case Dq: return launch_simt_bt<Dq>(BT, a);
    switch (DP4) {
        FD_CASE(1) FD_CASE(2) FD_CASE(3) FD_CASE(4) FD_CASE(5) FD_CASE(6) FD_CASE(7) FD_CASE(8)
        default: return false;
    }
#undef FD_CASE
}

int pick_bt(int bc) { return bc <= 4 ? 4 : bc <= 8 ? 8 : bc <= 16 ? 16 : 32; }

}  // namespace

}  // namespace fd

// ================================================================================================
// fd_apply_general_static: the split direct-difference block product for callers that cannot
// allocate device memory.
//
// Some hosts of this library hold no allocator they may call at the point where they need a
// kernel product: code running inside another framework's stream callback or capture-adjacent
// region, a plug-in that is handed input and output buffers only, a process whose memory pool
// is owned and sized by someone else.  For them every byte of scratch the ordinary entry points
// take from the caller's workspace lives here instead, in one file-scope device array of fixed
// size that each GPU loading the library keeps until the process exits.
//
// Scratch layout inside the array (floats): padded copy of the points, packed right-hand block,
// split-column partial sums.  Nothing in it has to start at zero: every word a launch reads was
// written earlier in the same call.  All calls share the array, so two calls that overlap on the
// GPU (different streams, or different host threads) race; serialise them.
namespace fd {
namespace {

constexpr size_t kStaticXs = (size_t)FD_STATIC_MAX_N * FD_STATIC_MAX_D;          // padded points
constexpr size_t kStaticWp = (size_t)FD_STATIC_MAX_N * FD_STATIC_MAX_B;          // packed right block
constexpr size_t kStaticPart = (size_t)3 << 19;                                  // split partials (6 MiB)
constexpr size_t kStaticFloats = kStaticXs + kStaticWp + kStaticPart;            // 8 MiB in total

static __device__ __align__(256) float g_static_scratch[kStaticFloats];

// Device address of the array per device ordinal, resolved on the first call made with that device current.
// (In host code the symbol's name is only a handle; the address a kernel can use comes from the runtime.)
constexpr int kMaxDevices = 64;
float* g_static_ptr[kMaxDevices] = {};

__global__ void k_static_pad_copy(const float* __restrict__ src, int64_t ld, int64_t n, int D, int DP, float* __restrict__ dst) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t total = n * DP;
    for (; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx / DP;
        const int k = (int)(idx - i * DP);
        dst[idx] = k < D ? src[i * ld + k] : 0.0f;
    }
}

fd_status static_fail(char* errbuf, size_t errlen, fd_status st, const char* fmt, long long a = 0, long long b = 0) {
    if (errbuf && errlen) snprintf(errbuf, errlen, fmt, a, b);
    return st;
}

}  // namespace
}  // namespace fd

extern "C" fd_status fd_apply_general_static(const float* X_dev, int64_t N, int32_t D, int64_t ldx, double beta,
                                             const float* left_dev, const float* right_dev, const float* V_dev,
                                             int64_t ldv, int32_t b, float* Y_dev, int64_t ldy, void* cuda_stream,
                                             char* errbuf, size_t errbuf_len) {
    using namespace fd;
    if (errbuf && errbuf_len) errbuf[0] = 0;
    if (!X_dev || !V_dev || !Y_dev) return static_fail(errbuf, errbuf_len, FD_ERR_INVALID, "X, V and Y must be non-null");
    if (N < 1 || D < 1 || b < 1 || ldx < D || ldv < N || ldy < N || !(beta > 0) || !(beta < 1e30))
        return static_fail(errbuf, errbuf_len, FD_ERR_INVALID, "bad size, pitch or beta");
    if (N > FD_STATIC_MAX_N) return static_fail(errbuf, errbuf_len, FD_ERR_UNSUPPORTED, "N = %lld exceeds FD_STATIC_MAX_N = %lld", (long long)N, FD_STATIC_MAX_N);
    if (D > FD_STATIC_MAX_D) return static_fail(errbuf, errbuf_len, FD_ERR_UNSUPPORTED, "D = %lld exceeds FD_STATIC_MAX_D = %lld", D, FD_STATIC_MAX_D);
    if (b > FD_STATIC_MAX_B) return static_fail(errbuf, errbuf_len, FD_ERR_UNSUPPORTED, "b = %lld exceeds FD_STATIC_MAX_B = %lld", b, FD_STATIC_MAX_B);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);

    // set-up, once per device: resolve the device address of the scratch array
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return static_fail(errbuf, errbuf_len, FD_ERR_CUDA, "cudaGetDevice failed or device ordinal out of range");
    if (!g_static_ptr[dev]) {
        float* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress((void**)&ptr, g_static_scratch);
        if (e != cudaSuccess || !ptr) return static_fail(errbuf, errbuf_len, FD_ERR_CUDA, "cudaGetSymbolAddress failed (%lld)", (long long)e);
        g_static_ptr[dev] = ptr;
    }
    float* xs = g_static_ptr[dev];
    float* wp = xs + kStaticXs;
    float* part = wp + kStaticWp;

    const int DP = (int)round_up(D, 4), DP4 = DP / 4;
    const int BT = pick_bt(b);
    const float nbeta2 = (float)(-beta * kLog2e);
    int grid_copy = (int)ceil_div(N * DP, 256);
    k_static_pad_copy<<<grid_copy, 256, 0, stream>>>(X_dev, ldx, N, D, DP, xs);
    ++g_launches;
    dim3 pg((unsigned)ceil_div(N, 32), (unsigned)ceil_div(BT, 32));
    k_pack_w<<<pg, dim3(32, 8), 0, stream>>>(V_dev, ldv, right_dev, N, 0, b, BT, wp);
    ++g_launches;
    // split the column range so that ~600 CTAs run, within the partials' capacity
    const int64_t row_tiles = ceil_div(N, kRows);
    int64_t sp = row_tiles >= 592 ? 1 : ceil_div(592, row_tiles);
    const int64_t cap = (int64_t)(kStaticPart / ((size_t)BT * (size_t)N));
    if (sp > cap) sp = cap;
    if (sp > ceil_div(N, kTJ)) sp = ceil_div(N, kTJ);
    if (sp < 1) sp = 1;
    const int64_t jps = round_up(ceil_div(N, sp), kTJ);
    sp = ceil_div(N, jps);
    dim3 grid((unsigned)row_tiles, (unsigned)sp);
    bool ok;
    if (sp == 1) {
        ok = launch_simt_any(DP4, BT, SimtArgs{grid, stream, xs, N, nbeta2, wp, jps, left_dev, Y_dev, ldy, 0, b});
        ++g_launches;
    } else {
        ok = launch_simt_any(DP4, BT, SimtArgs{grid, stream, xs, N, nbeta2, wp, jps, nullptr, part, N, (int64_t)BT * N, BT});
        ++g_launches;
        if (ok) {
            dim3 rg((unsigned)ceil_div(N, 256), (unsigned)b);
            k_reduce_block<<<rg, 256, 0, stream>>>(part, (int)sp, (int64_t)BT * N, N, b, left_dev, Y_dev, ldy);
            ++g_launches;
        }
    }
    if (!ok) return static_fail(errbuf, errbuf_len, FD_ERR_UNSUPPORTED, "no kernel instantiation for this D, b");
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return static_fail(errbuf, errbuf_len, FD_ERR_CUDA, "kernel launch failed (%lld)", (long long)e);
    return FD_OK;
}
