// O(N D) set-up: padded copy of the points, fp64 column means, mean and max of |x - mu|^2
// (the statistic Eq. 7 needs), and the O(N) elementwise / reduction helpers of the degree pass.
#include <algorithm>
#include <cstring>

#include "fd_internal.h"

namespace fd {

namespace {

constexpr int kRedBlocks = 1024;

// dst[i * DP + k] = src[i * ld + keep[k]] for the kept coordinates, zero padding up to DP.
__global__ void k_pad_copy(const float* __restrict__ src, int64_t ld, int64_t n, const Coords co, int DP, float* __restrict__ dst) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t total = n * DP;
    for (; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = idx / DP;
        int k = (int)(idx - i * DP);
        dst[idx] = k < co.kept ? src[i * ld + co.keep[k]] : 0.0f;
    }
}

// Column sums, minima and maxima.  Threads run along the rows' contiguous storage (thread t: coordinate t % DP of every
// (256 / DP)-th row of the block's share), one partial result per block and coordinate.
__global__ void __launch_bounds__(256)
k_colsum_partial(const float* __restrict__ xs, int64_t n, int DP, double* __restrict__ part, float2* __restrict__ minmax) {
    __shared__ double s_sum[256];
    __shared__ float2 s_mm[256];
    const int groups = 256 / DP, k = threadIdx.x % DP, g = threadIdx.x / DP;
    double acc = 0.0;
    float lo = INFINITY, hi = -INFINITY;
    if (g < groups)
        for (int64_t i = (int64_t)blockIdx.x * groups + g; i < n; i += (int64_t)gridDim.x * groups) {
            const float v = xs[i * DP + k];
            acc += (double)v;
            lo = fminf(lo, v); hi = fmaxf(hi, v);
        }
    s_sum[threadIdx.x] = acc; s_mm[threadIdx.x] = make_float2(lo, hi);
    __syncthreads();
    if (g == 0) {
        for (int q = 1; q < groups; ++q) {
            acc += s_sum[q * DP + k];
            lo = fminf(lo, s_mm[q * DP + k].x); hi = fmaxf(hi, s_mm[q * DP + k].y);
        }
        part[(size_t)blockIdx.x * DP + k] = acc;
        minmax[(size_t)blockIdx.x * DP + k] = make_float2(lo, hi);
    }
}

// mu, and a mask of the coordinates that are not the same for all points (bit k; written as a double's bits to *varying).
__global__ void __launch_bounds__(1024)
k_colsum_final(const double* __restrict__ part, const float2* __restrict__ minmax, int blocks, int DP, int64_t n, int center, double* __restrict__ mu,
               unsigned long long* __restrict__ varying) {
    __shared__ double s_sum[16][64];
    __shared__ float2 s_mm[16][64];
    __shared__ unsigned int mask[2];
    const int k = threadIdx.x % 64, g = threadIdx.x / 64;
    double acc = 0.0;
    float lo = INFINITY, hi = -INFINITY;
    if (k < DP)
        for (int b = g; b < blocks; b += 16) {
            acc += part[(size_t)b * DP + k];
            const float2 m = minmax[(size_t)b * DP + k];
            lo = fminf(lo, m.x); hi = fmaxf(hi, m.y);
        }
    s_sum[g][k] = acc; s_mm[g][k] = make_float2(lo, hi);
    __syncthreads();
    if (g != 0) return;
    for (int q = 1; q < 16; ++q) {
        acc += s_sum[q][k];
        lo = fminf(lo, s_mm[q][k].x); hi = fmaxf(hi, s_mm[q][k].y);
    }
    if (k < DP) mu[k] = center ? acc / (double)n : 0.0;
    const unsigned int b = __ballot_sync(0xffffffffu, k < DP && !(lo == hi));
    if ((k & 31) == 0) mask[k / 32] = b;
    asm volatile("bar.sync 1, 64;" ::: "memory");
    if (k == 0) *varying = (unsigned long long)mask[0] | ((unsigned long long)mask[1] << 32);
}

// mu[k] = mu[keep[k]]
__global__ void k_compact_mu(double* __restrict__ mu, const Coords co, int DP) {
    __shared__ double t[64];
    if ((int)threadIdx.x < DP) t[threadIdx.x] = (int)threadIdx.x < co.kept ? mu[co.keep[threadIdx.x]] : 0.0;
    __syncthreads();
    if ((int)threadIdx.x < DP) mu[threadIdx.x] = t[threadIdx.x];
}

// extra[i] = squared distance of external row i from the points in the dropped coordinates (which all points share); per-block maxima.
__global__ void __launch_bounds__(256)
k_row_extra(const float* __restrict__ X, int64_t ld, int64_t n, const Coords co, double* __restrict__ extra, double* __restrict__ part_max) {
    __shared__ double s_max[256];
    double mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        double e = 0.0;
        for (int k = 0; k < co.dropped; ++k) { const double v = (double)X[i * ld + co.drop[k]] - (double)co.value[k]; e += v * v; }
        extra[i] = e;
        mx = e > mx || e != e ? e : mx;
    }
    s_max[threadIdx.x] = mx;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) { const double o = s_max[threadIdx.x + off]; if (o > s_max[threadIdx.x] || o != o) s_max[threadIdx.x] = o; }
        __syncthreads();
    }
    if (threadIdx.x == 0) part_max[blockIdx.x] = s_max[0];
}

// out[i] = left[i] exp(-beta extra[i])
__global__ void k_row_factor(const float* __restrict__ left, const double* __restrict__ extra, double beta, int64_t n, float* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)((left ? (double)left[i] : 1.0) * exp(-beta * extra[i]));
}

// Per block: sum and max over its rows of |x_i - mu|^2 in fp64.
__global__ void k_sqnorm_partial(const float* __restrict__ xs, int64_t n, int DP, const double* __restrict__ mu,
                                 double* __restrict__ part_sum, double* __restrict__ part_max) {
    __shared__ double s_sum[256];
    __shared__ double s_max[256];
    double acc = 0.0, mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double r = 0.0;
        for (int k = 0; k < DP; ++k) {
            double v = (double)xs[i * DP + k] - mu[k];
            r += v * v;
        }
        acc += r;
        mx = r > mx ? r : mx;
    }
    s_sum[threadIdx.x] = acc; s_max[threadIdx.x] = mx;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) {
            s_sum[threadIdx.x] += s_sum[threadIdx.x + off];
            double o = s_max[threadIdx.x + off];
            if (o > s_max[threadIdx.x]) s_max[threadIdx.x] = o;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { part_sum[blockIdx.x] = s_sum[0]; part_max[blockIdx.x] = s_max[0]; }
}

__global__ void k_pow(const float* __restrict__ in, double p, float* __restrict__ out, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        // fp64 for the power: O(N) work, and s feeds every later product
        out[i] = (float)pow((double)in[i], p);
    }
}

// s = qa * d^-1/2 (qa null: 1), and copies of q, d, s where they are wanted.
__global__ void k_scale_vec(const float* __restrict__ qa, const float* __restrict__ q, const float* __restrict__ d, float* __restrict__ s, int64_t n,
                            float* __restrict__ q_out, float* __restrict__ d_out, float* __restrict__ s_out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float di = d[i], v = (float)((qa ? (double)qa[i] : 1.0) / sqrt((double)di));
    s[i] = v;
    if (q_out) q_out[i] = q[i];
    if (d_out) d_out[i] = di;
    if (s_out) s_out[i] = v;
}

// Stage 1: block partial sums (fixed assignment of elements to threads -> deterministic).
__global__ void k_sum_partial(const float* __restrict__ q, const double* __restrict__ rowsq, int64_t n,
                              double* __restrict__ part) {
    __shared__ double s_a[256];
    __shared__ double s_b[256];
    double a = 0.0, b = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        a += (double)q[i];
        if (rowsq) b += rowsq[i];
    }
    s_a[threadIdx.x] = a; s_b[threadIdx.x] = b;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) { s_a[threadIdx.x] += s_a[threadIdx.x + off]; s_b[threadIdx.x] += s_b[threadIdx.x + off]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { part[2 * blockIdx.x] = s_a[0]; part[2 * blockIdx.x + 1] = s_b[0]; }
}

// Fixed order: 256 strided sums, then a tree.
__global__ void __launch_bounds__(256)
k_sum_final(const double* __restrict__ part, int blocks, double* __restrict__ out) {
    __shared__ double s_a[256], s_b[256];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < blocks; i += 256) { a += part[2 * i]; b += part[2 * i + 1]; }
    s_a[threadIdx.x] = a; s_b[threadIdx.x] = b;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) { s_a[threadIdx.x] += s_a[threadIdx.x + off]; s_b[threadIdx.x] += s_b[threadIdx.x + off]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { out[0] = s_a[0]; out[1] = s_b[0]; }
}

__global__ void k_scale_cols_pow(const float* __restrict__ v, int64_t ldv, int cols, const float* __restrict__ d, double p,
                                 float* __restrict__ out, int64_t ldout, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float f = (float)pow((double)d[i], p);
    for (int c = 0; c < cols; ++c) out[i + (int64_t)c * ldout] = v[i + (int64_t)c * ldv] * f;
}

inline int grid_for(int64_t n, int block, int cap = 65535 * 8) {
    int64_t g = ceil_div(n, block);
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

fd_status setup_points(fd_ctx* c, const float* X_dev, int64_t ldx) {
    Layout& L = c->L;
    const int64_t N = L.N;
    Coords& co = c->coords;
    co.kept = L.D; co.dropped = 0;
    for (int k = 0; k < L.D; ++k) co.keep[k] = (uint8_t)k;
    k_pad_copy<<<grid_for(N * L.DP, 256, 148 * 16), 256, 0, c->stream>>>(X_dev, ldx, N, co, L.DP, c->xs());
    FD_LAUNCH_CHECK(c, "k_pad_copy");
    double* mu = c->at<double>(L.mu);
    double* sums = c->at<double>(L.sums);
    // partial results: one per block and coordinate (scratch: the Gram-form operand buffers, at least 16 KB per K slab)
    double* part = c->at<double>(L.xp_col);
    float2* minmax = c->at<float2>(L.xp_row);
    const int64_t room = L.NP * L.K16 * 64 / (8 * L.DP);
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(room, 592), ceil_div(N, 256 / L.DP)));
    k_colsum_partial<<<blocks, 256, 0, c->stream>>>(c->xs(), N, L.DP, part, minmax);
    FD_LAUNCH_CHECK(c, "k_colsum_partial");
    k_colsum_final<<<1, 1024, 0, c->stream>>>(part, minmax, blocks, L.DP, N, c->centered, mu, reinterpret_cast<unsigned long long*>(sums + 2048));
    FD_LAUNCH_CHECK(c, "k_colsum_final");
    int nb = grid_for(N, 256, 512);
    k_sqnorm_partial<<<nb, 256, 0, c->stream>>>(c->xs(), N, L.DP, mu, sums, sums + 1024);
    FD_LAUNCH_CHECK(c, "k_sqnorm_partial");
    double host[2049];
    FD_CUDA(c, cudaMemcpyAsync(host, sums, sizeof host, cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    double tot = 0.0, mx = 0.0;
    for (int i = 0; i < nb; ++i) { tot += host[i]; if (host[1024 + i] > mx) mx = host[1024 + i]; }
    if (!(tot == tot) || !(tot < 1e300)) return fail(c, FD_ERR_NONFINITE, "non-finite input points");
    c->mean_sq = tot / (double)N;
    c->max_sq = mx;
    // Coordinates that all points share (zero padding, a frozen degree of freedom) add nothing to any distance between them: where
    // leaving them out saves padded coordinates, the kernels work on the others alone.  External rows keep their
    // distance in the dropped coordinates as a factor per row (stage_rows).  D = 32 with 20 zeros, N = 8192, b = 8: 200 -> 105 us a product.
    unsigned long long varying;
    std::memcpy(&varying, host + 2048, 8);
    Coords cut{};
    for (int k = 0; k < L.D; ++k) {
        if ((varying >> k) & 1) cut.keep[cut.kept++] = (uint8_t)k;
        else cut.drop[cut.dropped++] = (uint8_t)k;
    }
    if (cut.kept == 0) { cut.keep[0] = cut.drop[--cut.dropped]; cut.kept = 1; }
    const int DP = (int)round_up(cut.kept, 4);
    if (DP >= L.DP) return FD_OK;
    float first[64];
    FD_CUDA(c, cudaMemcpyAsync(first, X_dev, sizeof(float) * (size_t)L.D, cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    for (int k = 0; k < cut.dropped; ++k) cut.value[k] = first[cut.drop[k]];
    co = cut;
    L.DP = DP;
    L.K16 = (int32_t)ceil_div(cut.kept + 4, 16);
    k_pad_copy<<<grid_for(N * L.DP, 256, 148 * 16), 256, 0, c->stream>>>(X_dev, ldx, N, co, L.DP, c->xs());
    FD_LAUNCH_CHECK(c, "k_pad_copy(kept)");
    k_compact_mu<<<1, 64, 0, c->stream>>>(mu, co, L.DP);
    FD_LAUNCH_CHECK(c, "k_compact_mu");
    // (X may be released after the call, as before: the copies above are complete)
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    return FD_OK;
}

fd_status stage_rows(fd_ctx* c, const float* Xrow_dev, int64_t ldxrow, int64_t r0, int64_t n) {
    const Layout& L = c->L;
    const float* X = Xrow_dev + r0 * ldxrow;
    k_pad_copy<<<grid_for(n * L.DP, 256, 148 * 16), 256, 0, c->stream>>>(X, ldxrow, n, c->coords, L.DP, c->at<float>(L.xrow));
    FD_LAUNCH_CHECK(c, "k_pad_copy(rows)");
    // largest |x - mu|^2 among the staged rows: the Gram-form kernel's exponent budget must hold for them too, and
    // external rows may lie further from the centre than any of the context's own points (scratch: split partials)
    double* part = c->at<double>(L.part);
    const int nb = grid_for(n, 256, 512);
    k_sqnorm_partial<<<nb, 256, 0, c->stream>>>(c->at<float>(L.xrow), n, L.DP, c->at<double>(L.mu), part, part + 1024);
    FD_LAUNCH_CHECK(c, "k_sqnorm_partial(rows)");
    const bool cut = c->coords.dropped > 0;
    if (cut) {
        k_row_extra<<<nb, 256, 0, c->stream>>>(X, ldxrow, n, c->coords, c->at<double>(L.rowsq), part + 2048);
        FD_LAUNCH_CHECK(c, "k_row_extra");
    }
    double host[2048 + 512];
    FD_CUDA(c, cudaMemcpyAsync(host, part, sizeof(double) * (size_t)(cut ? 2048 + 512 : 2048), cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    double tot = 0.0, mx = 0.0, ex = 0.0;
    for (int i = 0; i < nb; ++i) {
        tot += host[i];
        if (host[1024 + i] > mx) mx = host[1024 + i];
        if (cut) ex += host[2048 + i];
    }
    if (!(tot == tot) || !(tot < 1e300) || !(ex == ex) || !(ex < 1e300)) return fail(c, FD_ERR_NONFINITE, "non-finite row points");
    c->row_max_sq = mx;
    c->row_extra = ex > 0.0;
    return FD_OK;
}

fd_status row_factor(fd_ctx* c, const float* left, double beta, int64_t n, const float** out) {
    *out = left;
    if (!c->row_extra) return FD_OK;
    float* f = c->at<float>(c->L.symsum);                         // (the symmetric row sums never run between staging and product)
    k_row_factor<<<grid_for(n, 256), 256, 0, c->stream>>>(left, c->at<double>(c->L.rowsq), beta, n, f);
    FD_LAUNCH_CHECK(c, "k_row_factor");
    *out = f;
    return FD_OK;
}

fd_status ew_pow(fd_ctx* c, const float* in, double p, float* out, int64_t n) {
    k_pow<<<grid_for(n, 256), 256, 0, c->stream>>>(in, p, out, n);
    FD_LAUNCH_CHECK(c, "k_pow");
    return FD_OK;
}

fd_status ew_scale_vec(fd_ctx* c, const float* qa, const float* q, const float* d, float* s, int64_t n, float* q_out, float* d_out, float* s_out) {
    k_scale_vec<<<grid_for(n, 256), 256, 0, c->stream>>>(qa, q, d, s, n, q_out, d_out, s_out);
    FD_LAUNCH_CHECK(c, "k_scale_vec");
    return FD_OK;
}

fd_status reduce_sums(fd_ctx* c, const float* q, const double* rowsq, int64_t n, double* out_dev) {
    double* sums = c->at<double>(c->L.sums);
    int nb = grid_for(n, 256, kRedBlocks);
    k_sum_partial<<<nb, 256, 0, c->stream>>>(q, rowsq, n, sums);
    FD_LAUNCH_CHECK(c, "k_sum_partial");
    k_sum_final<<<1, 256, 0, c->stream>>>(sums, nb, out_dev);
    FD_LAUNCH_CHECK(c, "k_sum_final");
    return FD_OK;
}

fd_status scale_cols_by_pow(fd_ctx* c, const float* v, int64_t ldv, int32_t cols, const float* d, double p,
                            float* out, int64_t ldout, int64_t n) {
    k_scale_cols_pow<<<grid_for(n, 256), 256, 0, c->stream>>>(v, ldv, cols, d, p, out, ldout, n);
    FD_LAUNCH_CHECK(c, "k_scale_cols_pow");
    return FD_OK;
}

}  // namespace fd
