// Tall-skinny dense kernels for the eigensolver (O(N m b) work around the quadratic apply): A^T B with fp64 accumulation and a
// deterministic two-stage reduction, C = A S updates, column copies.  All blocks are column-major with N rows; a left
// (right) factor may consist of two column ranges that lie in different arrays.
//
// What bounds them: FMA issue at N = 2^17 and up (one N x 200 x 32 product is 0.84 G FMAs = 24 us at the measured 124 FFMA per clock
// per SM, its panel 105 MB = 16 us of HBM), launch and memory latency at N = 2^14.
#include <algorithm>

#include "fd_dense.h"

namespace fd {

namespace {

constexpr int kTnRows = 32;       // rows per pipeline stage
constexpr int kTnPitch = 36;      // floats between two columns of a stage: 16-byte reads of 8 neighbouring columns hit all 32 banks
constexpr int kTnStages = 3;
constexpr int kTnFlush = 2;       // stages summed in fp32 (64 terms) before the sums are added in fp64

__device__ __forceinline__ const float* panel_col(const Panel& a, int c) {
    return c < a.m1 ? a.p1 + (int64_t)c * a.ld : a.p2 + (int64_t)(c - a.m1) * a.ld;
}
// Copies 4 consecutive rows of a column into shared memory; rows at or beyond `valid` (0..4) read as zero.
template <bool ALIGNED>
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, int valid) {
    if (ALIGNED) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(4 * valid) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * i), "l"(src + (i < valid ? i : 0)), "r"(i < valid ? 4 : 0) : "memory");
    }
}

// part[chunk][i + j * m] = sum over this chunk's rows of A[r, i] * B[r, j] for a tile of 16 UI x 8 UJ outputs.
// 128 threads; thread (ti, tj) owns columns ti + 16 u of A and tj + 8 v of B.  Stages keep the columns contiguous (no transpose: a
// stage is filled by asynchronous copies), a thread reads four rows of a column at once, so 4 UI UJ FMAs follow UI + UJ
// 16-byte reads.  Products of 64 consecutive rows are accumulated in fp32 (entries of orthonormal columns are ~N^-1/2, so a
// 64-term partial sum loses ~1e-10 absolute) and every such partial sum is added to an fp64 accumulator, which keeps the
// long sum over N rows at fp64 accuracy at fp32 FMA speed.
// N = 2^17, 200 x 32: 55 us against 106 for 4 x 4 outputs a thread from transposed stages without copies in flight.
template <int UI, int UJ, bool ALIGNED>
__global__ void __launch_bounds__(128)
k_tn_partial(const Panel A, const Panel B, int64_t N, int64_t rows_per_chunk, double* __restrict__ part) {
    grid_go();
    extern __shared__ __align__(16) float sm[];
    constexpr int TI = 16 * UI, TJ = 8 * UJ, kStage = (TI + TJ) * kTnPitch;
    const int m = A.m1 + A.m2, n = B.m1 + B.m2;
    const int ti0 = blockIdx.x * TI, tj0 = blockIdx.y * TJ;
    const int64_t r_beg = (int64_t)blockIdx.z * rows_per_chunk;
    const int64_t r_end = r_beg + rows_per_chunk < N ? r_beg + rows_per_chunk : N;
    const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
    const int steps = (int)((r_end - r_beg + kTnRows - 1) / kTnRows);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);

    auto load = [&](int s) {
        if (s < steps) {
            const int64_t r0 = r_beg + (int64_t)s * kTnRows;
            const uint32_t st = sbase + 4u * (uint32_t)((s % kTnStages) * kStage);
            // eight threads copy the 32 rows of a column
            for (int t = threadIdx.x; t < (TI + TJ) * (kTnRows / 4); t += 128) {
                const int cc = t >> 3, rr = (t & 7) * 4;
                const bool left = cc < TI;
                const int col = left ? ti0 + cc : tj0 + cc - TI;
                int64_t valid = r_end - (r0 + rr);
                valid = valid < 0 ? 0 : valid > 4 ? 4 : valid;
                if (col >= (left ? m : n)) valid = 0;
                const float* src = left ? panel_col(A, col < m ? col : 0) : panel_col(B, col < n ? col : 0);
                copy4<ALIGNED>(st + 4u * (uint32_t)(cc * kTnPitch + rr), src + (valid > 0 ? r0 + rr : 0), (int)valid);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    double acc[UI][UJ];
    float f[UI][UJ];
#pragma unroll
    for (int u = 0; u < UI; ++u)
#pragma unroll
        for (int v = 0; v < UJ; ++v) { acc[u][v] = 0.0; f[u][v] = 0.f; }
#pragma unroll
    for (int s = 0; s < kTnStages - 1; ++s) load(s);
    for (int s = 0; s < steps; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kTnStages - 2) : "memory");
        __syncthreads();                               // stage s has landed; everybody is done with the stage that load() refills
        load(s + kTnStages - 1);
        const float* st = sm + (s % kTnStages) * kStage;
        const float* sa = st + ti * kTnPitch;
        const float* sb = st + (TI + tj) * kTnPitch;
#pragma unroll 4
        for (int rr = 0; rr < kTnRows; rr += 4) {
            float4 a[UI], b[UJ];
#pragma unroll
            for (int u = 0; u < UI; ++u) a[u] = *reinterpret_cast<const float4*>(sa + 16 * u * kTnPitch + rr);
#pragma unroll
            for (int v = 0; v < UJ; ++v) b[v] = *reinterpret_cast<const float4*>(sb + 8 * v * kTnPitch + rr);
#pragma unroll
            for (int u = 0; u < UI; ++u)
#pragma unroll
                for (int v = 0; v < UJ; ++v) {
                    float x = fmaf(a[u].x, b[v].x, f[u][v]);
                    x = fmaf(a[u].y, b[v].y, x);
                    x = fmaf(a[u].z, b[v].z, x);
                    f[u][v] = fmaf(a[u].w, b[v].w, x);
                }
        }
        if (s % kTnFlush == kTnFlush - 1 || s + 1 == steps) {
#pragma unroll
            for (int u = 0; u < UI; ++u)
#pragma unroll
                for (int v = 0; v < UJ; ++v) { acc[u][v] += (double)f[u][v]; f[u][v] = 0.f; }
        }
    }
    double* o = part + (size_t)blockIdx.z * m * n;
#pragma unroll
    for (int u = 0; u < UI; ++u)
#pragma unroll
        for (int v = 0; v < UJ; ++v) {
            const int i = ti0 + ti + 16 * u, j = tj0 + tj + 8 * v;
            if (i < m && j < n) o[i + (size_t)j * m] = acc[u][v];
        }
}

// out[e] = sum of the chunks' partials in a fixed order: 32 outputs x 8 partial sums per block, so that the chunks are read in
// parallel.  `out` may be page-locked host memory: the values are stored there directly, no copy follows.
__global__ void __launch_bounds__(256)
k_tn_reduce(const double* __restrict__ part, int chunks, int64_t mm, double* __restrict__ out) {
    grid_wait();
    grid_go();
    __shared__ double sm[8][33];
    const int64_t e = (int64_t)blockIdx.x * 32 + threadIdx.x;
    double a0 = 0.0, a1 = 0.0;
    if (e < mm) {
        int c = threadIdx.y;
        for (; c + 8 < chunks; c += 16) { a0 += part[(size_t)c * mm + e]; a1 += part[(size_t)(c + 8) * mm + e]; }
        if (c < chunks) a0 += part[(size_t)c * mm + e];
    }
    sm[threadIdx.y][threadIdx.x] = a0 + a1;
    __syncthreads();
    if (threadIdx.y == 0 && e < mm) {
        double acc = 0.0;
#pragma unroll
        for (int y = 0; y < 8; ++y) acc += sm[y][threadIdx.x];
        out[e] = acc;
    }
}

// C[i, c] = sum_k A[i, k] S[k, c] for a strip of PT columns; RPT rows per thread (two where there are enough rows: half the
// shared-memory reads per FMA).  S is staged 32 rows at a time; the rows of A are read straight from memory, eight columns in flight.
// N = 2^17, m = 200, p = 32: 48 us against 91 with one row per thread and four loads in flight.
// KS groups of 128 threads share the columns of A (partial sums meet in shared memory): few rows leave each thread a long chain of dependent
// loads otherwise (N = 16384, m = 260, p = 41: 27 -> 14 us with four groups).
template <int PT, int RPT, int KS>
__global__ void __launch_bounds__(128 * KS)
k_nn(const Panel A, const float* __restrict__ S, int lds, int p, float* __restrict__ C, int64_t ldc, int64_t N) {
    grid_wait();
    grid_go();
    static_assert(KS == 1 || RPT == 1, "split columns with one row per thread only");
    constexpr int kS = 32 * PT, kRed = KS > 1 ? (KS - 1) * PT * 128 : 0;
    __shared__ __align__(16) float smem[KS * kS > kRed ? KS * kS : kRed];
    const int m = A.m1 + A.m2;
    const int grp = threadIdx.x / 128, tid = threadIdx.x % 128;
    float* ss = smem + grp * kS;
    const int64_t i0 = (int64_t)blockIdx.x * (128 * RPT) + tid;
    const int c0 = blockIdx.y * PT;
    int64_t row[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) row[r] = i0 + 128 * r < N ? i0 + 128 * r : N - 1;
    float acc[RPT][PT];
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
        for (int c = 0; c < PT; ++c) acc[r][c] = 0.f;
    for (int kb0 = 0; kb0 < m; kb0 += 32 * KS) {
        const int k0 = kb0 + 32 * grp;                             // this group's 32 columns
        __syncthreads();
        for (int t = tid; t < 32 * PT; t += 128) {
            const int kk = t % 32, cc = t / 32;
            ss[kk * PT + cc] = (k0 + kk < m && c0 + cc < p) ? S[(k0 + kk) + (size_t)(c0 + cc) * lds] : 0.f;
        }
        __syncthreads();
        const int kn = m - k0 < 32 ? m - k0 : 32;
        for (int kb = 0; kb < kn; kb += 8) {
            float a[8][RPT];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = k0 + kb + u < m ? k0 + kb + u : m - 1;       // (padding columns meet zeros in S)
                const float* col = panel_col(A, k);
#pragma unroll
                for (int r = 0; r < RPT; ++r) a[u][r] = col[row[r]];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int c4 = 0; c4 < PT / 4; ++c4) {
                    const float4 s4 = *reinterpret_cast<const float4*>(&ss[(kb + u) * PT + 4 * c4]);
#pragma unroll
                    for (int r = 0; r < RPT; ++r) {
                        acc[r][4 * c4 + 0] = fmaf(a[u][r], s4.x, acc[r][4 * c4 + 0]);
                        acc[r][4 * c4 + 1] = fmaf(a[u][r], s4.y, acc[r][4 * c4 + 1]);
                        acc[r][4 * c4 + 2] = fmaf(a[u][r], s4.z, acc[r][4 * c4 + 2]);
                        acc[r][4 * c4 + 3] = fmaf(a[u][r], s4.w, acc[r][4 * c4 + 3]);
                    }
                }
        }
    }
    if (KS > 1) {
        __syncthreads();
        if (grp > 0) {
#pragma unroll
            for (int c = 0; c < PT; ++c) smem[((grp - 1) * PT + c) * 128 + tid] = acc[0][c];
        }
        __syncthreads();
        if (grp > 0) return;
#pragma unroll
        for (int q = 0; q < KS - 1; ++q)
#pragma unroll
            for (int c = 0; c < PT; ++c) acc[0][c] += smem[(q * PT + c) * 128 + tid];
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r)
        if (i0 + 128 * r < N) {
#pragma unroll
            for (int c = 0; c < PT; ++c)
                if (c0 + c < p) C[i0 + 128 * r + (int64_t)(c0 + c) * ldc] = acc[r][c];
        }
}

// dst[:, c] = src[:, idx[c]]
struct ColumnList { int n; uint16_t idx[256]; };
__global__ void k_gather_cols(const float* __restrict__ src, float* __restrict__ dst, int64_t ld, const ColumnList list, int64_t N) {
    grid_wait();
    grid_go();
    const int c = blockIdx.y;
    const float* s = src + (int64_t)list.idx[c] * ld;
    float* d = dst + (int64_t)c * ld;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) d[i] = s[i];
}

// out[c] = sum_i A[i, c]^2 in fp64; one block per column, fixed summation order (bit-reproducible).
__global__ void __launch_bounds__(1024)
k_col_sqnorms(const float* __restrict__ A, int64_t lda, int64_t N, double* __restrict__ out) {
    grid_wait();
    grid_go();
    __shared__ double sm[1024];
    const float* col = A + (int64_t)blockIdx.x * lda;
    double acc = 0.0;
    for (int64_t i0 = 0; i0 < N; i0 += 1024 * 8) {
        float f = 0.f;                               // 8 squares in fp32, then into the fp64 accumulator
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t i = i0 + (int64_t)u * 1024 + threadIdx.x;
            if (i < N) { const float v = col[i]; f = fmaf(v, v, f); }
        }
        acc += (double)f;
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int off = 512; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) sm[threadIdx.x] += sm[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sm[0];
}

// Counter-based uniform(-1, 1) fill for cold-start blocks (hash of (seed, element index)).
__global__ void k_random_fill(float* __restrict__ A, int64_t lda, int p, int64_t N, int64_t row0, uint32_t seed) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    for (int c = 0; c < p; ++c) {
        uint64_t z = (uint64_t)(i + row0) * 0x9E3779B97F4A7C15ull + ((uint64_t)(c + 1) << 40) + seed;
        z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ull; z ^= z >> 27; z *= 0x94D049BB133111EBull; z ^= z >> 31;
        A[i + (int64_t)c * lda] = (float)((double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0);
    }
}

__global__ void k_sqrt_vec(const float* __restrict__ d, float* __restrict__ out, int64_t N) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) out[i] = (float)sqrt((double)d[i]);
}

}  // namespace

namespace {

bool panel_aligned(const Panel& a) {
    return a.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(a.p1) & 15) == 0 && (a.m2 == 0 || (reinterpret_cast<uintptr_t>(a.p2) & 15) == 0);
}

template <int UI, int UJ, bool ALIGNED>
fd_status launch_tn(fd_ctx* c, const Panel& A, const Panel& B, int64_t N, int64_t max_chunks, double* scratch, int* chunks_out) {
    constexpr int TI = 16 * UI, TJ = 8 * UJ, smem = kTnStages * (TI + TJ) * kTnPitch * 4;
    const int m = A.m1 + A.m2, n = B.m1 + B.m2;
    // row chunks: two blocks per SM, at least two pipeline fills of rows each
    const int64_t tiles = ceil_div(m, TI) * ceil_div(n, TJ);
    int64_t chunks = std::max<int64_t>(1, (int64_t)c->sm_count * 2 / tiles);
    chunks = std::min(chunks, std::min(max_chunks, ceil_div(N, 2 * kTnRows)));
    const int64_t rpc = round_up(ceil_div(N, chunks), 2 * kTnRows);
    chunks = ceil_div(N, rpc);
    FD_CUDA(c, cudaFuncSetAttribute(k_tn_partial<UI, UJ, ALIGNED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const dim3 grid((unsigned)ceil_div(m, TI), (unsigned)ceil_div(n, TJ), (unsigned)chunks);
    // (not behind the kernel before: two blocks per SM, evenly)
    k_tn_partial<UI, UJ, ALIGNED><<<grid, 128, smem, c->stream>>>(A, B, N, rpc, scratch);
    FD_LAUNCH_CHECK(c, "k_tn_partial");
    *chunks_out = (int)chunks;
    return FD_OK;
}

}  // namespace

fd_status tn_product(fd_ctx* c, const Panel& A, const Panel& B, int64_t N, double* out, double* scratch, size_t scratch_doubles) {
    const int m = A.m1 + A.m2, n = B.m1 + B.m2;
    if (m < 1 || n < 1) return FD_OK;
    const size_t mm = (size_t)m * n;
    int chunks = 0;                                               // a rank that owns no rows contributes zeros
    if (N >= 1) {
        const int64_t max_chunks = (int64_t)std::min<size_t>(scratch_doubles / mm, 65535);
        if (max_chunks < 1) return fail(c, FD_ERR_WORKSPACE, "projection scratch too small for %d x %d", m, n);
        const bool al = panel_aligned(A) && panel_aligned(B);
        // tile heights 128 / 64 by the number of left columns, widths 32 / 16 by the number of right columns: padding columns cost
        // as much as real ones
#define FD_TN(UI, UJ) FD_TRY((al ? launch_tn<UI, UJ, true>(c, A, B, N, max_chunks, scratch, &chunks)                  \
                                 : launch_tn<UI, UJ, false>(c, A, B, N, max_chunks, scratch, &chunks)))
        if (m > 64) { if (n > 16) FD_TN(8, 4); else FD_TN(8, 2); }
        else { if (n > 16) FD_TN(4, 4); else FD_TN(4, 2); }
#undef FD_TN
    }
    FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)ceil_div((int64_t)mm, 32)), dim3(32, 8), 0, k_tn_reduce, (const double*)scratch, chunks, (int64_t)mm, out));
    FD_LAUNCH_CHECK(c, "k_tn_reduce");
    return FD_OK;
}

fd_status nn_product(fd_ctx* c, const Panel& A, const float* S_dev, int lds, int p, float* C, int64_t ldc, int64_t N) {
    if (p < 1 || N < 1) return FD_OK;
    if (A.m1 + A.m2 < 1) return fail(c, FD_ERR_INVALID, "nn_product: no columns");
    // strips of 32 columns and two rows per thread where that still gives every SM a few blocks, else strips of 32 / 16 / 8 columns
    // (the narrowest that holds p, at most 16: more blocks) with the columns of A shared by four groups of threads
    const unsigned rb = (unsigned)ceil_div(N, 128);
    if (p > 16 && ceil_div(N, 256) * ceil_div(p, 32) >= 3 * c->sm_count)
        FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)ceil_div(N, 256), (unsigned)ceil_div(p, 32)), dim3(128), 0, k_nn<32, 2, 1>, A, S_dev, lds, p, C, ldc, N));
    else if (p > 16 && rb * ceil_div(p, 32) >= 4 * c->sm_count)
        FD_CUDA(c, launch_behind(c->stream, dim3(rb, (unsigned)ceil_div(p, 32)), dim3(128), 0, k_nn<32, 1, 1>, A, S_dev, lds, p, C, ldc, N));
    else if (p > 8)
        FD_CUDA(c, launch_behind(c->stream, dim3(rb, (unsigned)ceil_div(p, 16)), dim3(512), 0, k_nn<16, 1, 4>, A, S_dev, lds, p, C, ldc, N));
    else
        FD_CUDA(c, launch_behind(c->stream, dim3(rb, 1u), dim3(512), 0, k_nn<8, 1, 4>, A, S_dev, lds, p, C, ldc, N));
    FD_LAUNCH_CHECK(c, "k_nn");
    return FD_OK;
}

fd_status gather_cols(fd_ctx* c, const float* src, float* dst, int64_t ld, const int* idx, int p, int64_t N) {
    if (p < 1 || N < 1) return FD_OK;
    if (p > 256) return fail(c, FD_ERR_INVALID, "gather_cols: more than 256 columns");
    ColumnList list;
    list.n = p;
    for (int i = 0; i < p; ++i) list.idx[i] = (uint16_t)idx[i];
    FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)std::min<int64_t>(64, ceil_div(N, 256)), (unsigned)p), dim3(256), 0, k_gather_cols, src, dst, ld, list, N));
    FD_LAUNCH_CHECK(c, "k_gather_cols");
    return FD_OK;
}

fd_status col_sqnorms(fd_ctx* c, const float* A, int64_t lda, int p, int64_t N, double* out) {
    if (p < 1) return FD_OK;
    FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)p), dim3(1024), 0, k_col_sqnorms, A, lda, N, out));
    FD_LAUNCH_CHECK(c, "k_col_sqnorms");
    return FD_OK;
}

fd_status random_fill(fd_ctx* c, float* A, int64_t lda, int p, int64_t N, int64_t row0, uint32_t seed) {
    if (N < 1 || p < 1) return FD_OK;
    k_random_fill<<<(unsigned)ceil_div(N, 256), 256, 0, c->stream>>>(A, lda, p, N, row0, seed);
    FD_LAUNCH_CHECK(c, "k_random_fill");
    return FD_OK;
}

fd_status sqrt_vec(fd_ctx* c, const float* d, float* out, int64_t N) {
    if (N < 1) return FD_OK;
    k_sqrt_vec<<<(unsigned)ceil_div(N, 256), 256, 0, c->stream>>>(d, out, N);
    FD_LAUNCH_CHECK(c, "k_sqrt_vec");
    return FD_OK;
}

fd_status copy_cols(fd_ctx* c, const float* src, int64_t lds, float* dst, int64_t ldd, int p, int64_t N) {
    if (p < 1 || N < 1) return FD_OK;
    FD_CUDA(c, cudaMemcpy2DAsync(dst, (size_t)ldd * 4, src, (size_t)lds * 4, (size_t)N * 4, (size_t)p,
                                 cudaMemcpyDeviceToDevice, c->stream));
    return FD_OK;
}

}  // namespace fd
