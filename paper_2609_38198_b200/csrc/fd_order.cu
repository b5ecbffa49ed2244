// Which tiles of the kernel matrix are zero, and the order of the points that makes whole tiles zero.
//
// A Gaussian kernel at a useful bandwidth is numerically zero for many pairs of points: beyond an exponent of 40 (base 2) both
// fp16 pieces of a kernel value are zero in the block product, beyond 60 its contribution to a degree sum is below the
// fixed-point unit.  With the points in the order in which they came every tile of 128 x 128 pairs holds some near pairs; with
// neighbours in consecutive positions tiles are compact and far tiles can be left out without changing the results.
//
// Coordinates: with more than 8 of them the tree and the boxes use the 8 leading principal directions of the samples (an orthogonal projection:
// distances there are lower bounds too), in which a low-dimensional data set's boxes are tight and cheap (R^30, N = 2^18: 65 %
// of the tiles remain instead of 73 % with boxes along the coordinates).
//
// Order: a k-d tree over 4096 sampled points (each node splits its samples at the median of their widest coordinate) down to leaves
// of about 128 points; all points are routed through it and sorted by leaf, stably.  It is made once per context, when a
// bandwidth first leaves at least 15 % of sampled pairs beyond the exponent, and costs about 0.6 ms at N = 2^18.  Vectors stay in
// the caller's order everywhere: the operand packing gathers through the permutation, the epilogues scatter.
//
// Lists: for a bandwidth and exponent limit, per row pair (256 points) the column tiles (128 points) whose bounding box comes
// close enough (distance of the two boxes: a lower bound for every pair).  Data that fill many dimensions (the
// 6-torus) have no far tiles; then the products run over all tiles as before.
// N = 2^18, R^30 on a two-dimensional manifold, beta = 2 (44 % of the pairs are not zero), both at the power limit: b = 32, 25.5 -> 20.1 ms a
// product; degree passes 23.2 -> 19.9 ms.
#include <algorithm>
#include <cmath>

#include "fd_dense.h"

namespace fd {

namespace {

constexpr int kSamples = 4096;

// Counts pairs of 1024 sampled points farther apart than limit2 (squared distance).
__global__ void __launch_bounds__(256)
k_far_pairs(const float* __restrict__ xs, int DP, int64_t n, float limit2, unsigned int* __restrict__ count) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;      // one sampled row per warp
    const float* xi = xs + (n * i / 1024) * DP;
    unsigned int far = 0;
    for (int j = lane; j < 1024; j += 32) {
        const float* xj = xs + (n * j / 1024) * DP;
        float d2 = 0.f;
        for (int k = 0; k < DP; ++k) { const float d = xi[k] - xj[k]; d2 = fmaf(d, d, d2); }
        far += d2 > limit2;
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) far += __shfl_xor_sync(0xffffffffu, far, m);
    if (lane == 0) atomicAdd(count, far);
}

// part[block][k * DP + l] = sum over this block's 128 samples of (x_k - mu_k) (x_l - mu_l).
__global__ void __launch_bounds__(256)
k_cov_partial(const float* __restrict__ xs, int DP, int64_t n, const double* __restrict__ mu, double* __restrict__ part) {
    extern __shared__ float sx[];                                  // 128 x DP
    for (int t = threadIdx.x; t < 128 * DP; t += 256) {
        const int64_t i = n * ((int64_t)blockIdx.x * 128 + t / DP) / kSamples;
        sx[t] = (float)((double)xs[i * DP + t % DP] - mu[t % DP]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < DP * DP; e += 256) {
        const int k = e / DP, l = e % DP;
        float a = 0.f;
        for (int r = 0; r < 128; ++r) a = fmaf(sx[r * DP + k], sx[r * DP + l], a);
        part[(size_t)blockIdx.x * DP * DP + e] = (double)a;
    }
}
__global__ void k_cov_sum(const double* __restrict__ part, int blocks, int n, double* __restrict__ out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double a = 0.0;
    for (int b = 0; b < blocks; ++b) a += part[(size_t)b * n + e];
    out[e] = a;
}
// z[i * 8 + c] = (x_i - mu) . dir_c
struct Directions { float v[8][64]; };
__global__ void __launch_bounds__(256)
k_project(const float* __restrict__ xs, int DP, int64_t n, const double* __restrict__ mu, const Directions dir, float* __restrict__ z) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    float a[8] = {};
    for (int k = 0; k < DP; ++k) {
        const float x = (float)((double)xs[i * DP + k] - mu[k]);
#pragma unroll
        for (int c = 0; c < 8; ++c) a[c] = fmaf(x, dir.v[c][k], a[c]);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) z[i * 8 + c] = a[c];
}

struct Node { int dim; float thr; };

// One level of the tree: block = node, its `len` samples are idx[node * len ..) (level 0: the sample itself).  Sorts them by the
// widest coordinate; the halves are the children.
__global__ void __launch_bounds__(512)
k_kd_level(const float* __restrict__ xs, int DP, int64_t n, int level, int* __restrict__ idx, Node* __restrict__ nodes) {
    __shared__ float key[kSamples];
    __shared__ int val[kSamples];
    __shared__ float s_lo[64], s_hi[64];
    __shared__ int s_dim;
    const int len = kSamples >> level, node = blockIdx.x;
    int* mine = idx + (size_t)node * len;
    for (int t = threadIdx.x; t < len; t += 512) val[t] = level == 0 ? (int)(n * t / kSamples) : mine[t];
    __syncthreads();
    // extent of every coordinate (a warp per coordinate)
    for (int k = threadIdx.x >> 5; k < DP; k += 16) {
        float lo = INFINITY, hi = -INFINITY;
        for (int t = threadIdx.x & 31; t < len; t += 32) { const float v = xs[(int64_t)val[t] * DP + k]; lo = fminf(lo, v); hi = fmaxf(hi, v); }
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m)); }
        if ((threadIdx.x & 31) == 0) { s_lo[k] = lo; s_hi[k] = hi; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int d = 0;
        for (int k = 1; k < DP; ++k)
            if (s_hi[k] - s_lo[k] > s_hi[d] - s_lo[d]) d = k;
        s_dim = d;
    }
    __syncthreads();
    const int dim = s_dim;
    for (int t = threadIdx.x; t < len; t += 512) key[t] = xs[(int64_t)val[t] * DP + dim];
    __syncthreads();
    for (int size = 2; size <= len; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < len / 2; t += 512) {
                const int a = 2 * t - (t & (stride - 1)), b = a + stride;
                const bool up = (a & size) == 0;
                const float ka = key[a], kb = key[b];
                const int va = val[a], vb = val[b];
                const bool gt = ka > kb || (ka == kb && va > vb);              // ties by index: the order is unique
                if (gt == up) { key[a] = kb; key[b] = ka; val[a] = vb; val[b] = va; }
            }
            __syncthreads();
        }
    for (int t = threadIdx.x; t < len; t += 512) mine[t] = val[t];
    if (threadIdx.x == 0) nodes[(1 << level) - 1 + node] = Node{dim, key[len / 2]};
}

// Leaf of every point, and how many points of each block of 1024 fall into each leaf (counts[leaf * blocks + block]).
__global__ void __launch_bounds__(1024)
k_kd_route(const float* __restrict__ xs, int DP, int64_t n, int depth, const Node* __restrict__ nodes, unsigned short* __restrict__ leaf,
           unsigned int* __restrict__ counts) {
    __shared__ unsigned int hist[kSamples];
    const int leaves = 1 << depth;
    for (int t = threadIdx.x; t < leaves; t += 1024) hist[t] = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    if (i < n) {
        int node = 0;
        for (int l = 0; l < depth; ++l) {
            const Node nd = nodes[(1 << l) - 1 + node];
            node = 2 * node + (xs[i * DP + nd.dim] >= nd.thr ? 1 : 0);
        }
        leaf[i] = (unsigned short)node;
        atomicAdd(&hist[node], 1u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < leaves; t += 1024) counts[(size_t)t * gridDim.x + blockIdx.x] = hist[t];
}
// Exclusive scan of each leaf's counts over the blocks (a warp per leaf); totals[leaf].
__global__ void __launch_bounds__(256)
k_leaf_scan(unsigned int* __restrict__ counts, int blocks, int leaves, unsigned int* __restrict__ totals) {
    const int leaf = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (leaf >= leaves) return;
    unsigned int* row = counts + (size_t)leaf * blocks;
    unsigned int base = 0;
    for (int b0 = 0; b0 < blocks; b0 += 32) {
        const unsigned int v = b0 + lane < blocks ? row[b0 + lane] : 0u;
        unsigned int s = v;
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) { const unsigned int o = __shfl_up_sync(0xffffffffu, s, m); if (lane >= m) s += o; }
        if (b0 + lane < blocks) row[b0 + lane] = base + s - v;
        base += __shfl_sync(0xffffffffu, s, 31);
    }
    if (lane == 0) totals[leaf] = base;
}
// out[i] = sum of in[0 .. i), out[n] = total (one block; in and out may not overlap).
__global__ void __launch_bounds__(1024)
k_scan(const unsigned int* __restrict__ in, int n, unsigned int* __restrict__ out) {
    __shared__ unsigned int s[1024];
    const int per = (n + 1023) / 1024, i0 = threadIdx.x * per;
    unsigned int sum = 0;
    for (int i = i0; i < min(n, i0 + per); ++i) sum += in[i];
    s[threadIdx.x] = sum;
    __syncthreads();
    for (int m = 1; m < 1024; m <<= 1) {
        const unsigned int o = (int)threadIdx.x >= m ? s[threadIdx.x - m] : 0u;
        __syncthreads();
        s[threadIdx.x] += o;
        __syncthreads();
    }
    unsigned int base = s[threadIdx.x] - sum;
    for (int i = i0; i < min(n, i0 + per); ++i) { out[i] = base; base += in[i]; }
    if (threadIdx.x == 1023) out[n] = s[1023];
}
// perm[position] = index, by leaf and in index order inside a leaf: the warps of a block take their turns.
__global__ void __launch_bounds__(1024)
k_scatter(const unsigned short* __restrict__ leaf, int64_t n, const unsigned int* __restrict__ counts, const unsigned int* __restrict__ base, int leaves,
          int* __restrict__ perm) {
    __shared__ unsigned int next[kSamples];
    for (int t = threadIdx.x; t < leaves; t += 1024) next[t] = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const unsigned int l = i < n ? leaf[i] : 0xffffu;
    const unsigned int peers = __match_any_sync(0xffffffffu, l);
    unsigned int rank = __popc(peers & ((1u << lane) - 1u));
    for (int w = 0; w < 32; ++w) {
        if ((int)(threadIdx.x >> 5) == w && i < n) {
            rank += next[l];
            __syncwarp(__activemask());
            if (lane == __ffs(peers) - 1) next[l] += __popc(peers);
        }
        __syncthreads();
    }
    if (i < n) perm[base[l] + counts[(size_t)l * gridDim.x + blockIdx.x] + rank] = (int)i;
}

// Bounding box of each tile of 128 consecutive positions: box[tile * 2 DP ..] = minima, then maxima.  Empty tiles get an empty box.
__global__ void __launch_bounds__(128)
k_boxes(const float* __restrict__ xs, int DP, int64_t n, const int* __restrict__ perm, float* __restrict__ box) {
    __shared__ float s_lo[4][64], s_hi[4][64];
    const int64_t p = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t i = p < n ? perm[p] : -1;
    for (int k = 0; k < DP; ++k) {
        const float v = i >= 0 ? xs[i * DP + k] : 0.f;
        float lo = i >= 0 ? v : INFINITY, hi = i >= 0 ? v : -INFINITY;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m)); }
        if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5][k] = lo; s_hi[threadIdx.x >> 5][k] = hi; }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < DP; k += 128) {
        box[(size_t)blockIdx.x * 2 * DP + k] = fminf(fminf(s_lo[0][k], s_lo[1][k]), fminf(s_lo[2][k], s_lo[3][k]));
        box[((size_t)blockIdx.x * 2 + 1) * DP + k] = fmaxf(fmaxf(s_hi[0][k], s_hi[1][k]), fmaxf(s_hi[2][k], s_hi[3][k]));
    }
}

// Column tiles of row pair blockIdx.x whose box comes within limit2 of the pair's box, ascending: list[pair * tiles ..]; counts[pair]
// of them, of which `upper[pair]` are tiles 2 pair and later (the symmetric row sums start there).
__global__ void __launch_bounds__(256)
k_lists(const float* __restrict__ box, int DP, int tiles, float limit2, unsigned short* __restrict__ list, unsigned int* __restrict__ counts,
        unsigned int* __restrict__ upper) {
    __shared__ float lo[64], hi[64];
    __shared__ unsigned int wsum[8];
    const int pair = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < DP; k += 256) {
        const float *a = box + (size_t)(2 * pair) * 2 * DP, *b = a + 2 * DP;
        lo[k] = fminf(a[k], b[k]); hi[k] = fmaxf(a[DP + k], b[DP + k]);
    }
    __syncthreads();
    unsigned int n = 0, below = 0;
    for (int t0 = 0; t0 < tiles; t0 += 256) {
        const int t = t0 + threadIdx.x;
        bool near = false;
        if (t < tiles) {
            const float* b = box + (size_t)t * 2 * DP;
            float d2 = 0.f;
            for (int k = 0; k < DP; ++k) {
                const float g = fmaxf(fmaxf(b[k] - hi[k], lo[k] - b[DP + k]), 0.f);
                d2 = fmaf(g, g, d2);
            }
            near = d2 <= limit2 || (t >> 1) == pair;                   // (an empty box is infinitely far; a pair's own tiles always count)
        }
        const unsigned int vote = __ballot_sync(0xffffffffu, near);
        if (lane == 0) wsum[warp] = __popc(vote);
        __syncthreads();
        unsigned int pos = n + __popc(vote & ((1u << lane) - 1u)), all = 0;
        for (int w = 0; w < 8; ++w) { if (w < warp) pos += wsum[w]; all += wsum[w]; }
        if (near) {
            list[(size_t)pair * tiles + pos] = (unsigned short)t;
            if (t == 2 * pair) below = pos + 1;                        // (one thread of the block sees it)
        }
        n += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) counts[pair] = n;
    if (below) upper[pair] = below - 1;
    __syncthreads();
    if (threadIdx.x == 0) upper[pair] = n - upper[pair];
}

}  // namespace

fd_status tile_lists(fd_ctx* c, double beta, int kind, bool decide) {
    const Layout& L = c->L;
    auto& st = c->lists[kind];
    if (L.perm == 0 || c->order_state < 0) return FD_OK;
    if (st.beta == beta && (!st.on || (c->listed_kind == kind && c->listed_beta == beta))) return FD_OK;
    // Beyond an exponent of 40 both fp16 pieces of a kernel value are zero (2^15 2^-40 = 2^-25 rounds to zero), beyond 60 a degree
    // contribution is below the fixed-point unit; the quarter covers the rounding of the boxes' distance.
    const double limit = kind == 0 ? 40.25 : 60.25;
    if (!decide && st.beta != beta) return FD_OK;
    const bool known = st.beta == beta;                            // decided before, only overwritten by the other kind's lists
    const int64_t N = L.N;
    const int tiles = (int)(L.NP / 128), pairs = (int)(L.NP / 256);
    const float limit2 = (float)(limit / (beta * kLog2e));
    if (!known) { st.on = false; st.beta = beta; }
    unsigned int* small = reinterpret_cast<unsigned int*>(c->at<char>(L.status) + 128);
    int* perm = c->at<int>(L.perm);
    float* box = c->at<float>(L.boxes);
    const bool project = L.DP > 8;
    const float* z = project ? c->at<float>(L.zproj) : c->xs();        // coordinates of the tree and the boxes
    const int ZP = project ? 8 : L.DP;
    if (!known && 4.0 * c->max_sq <= (double)limit2) return FD_OK;               // no two points are that far apart
    bool fresh = false;
    if (c->order_state == 0) {
        // (an order that left out too little at some bandwidth would leave out less at a smaller one: in units of the degree passes' limit)
        if (beta * (kind == 0 ? 60.25 / 40.25 : 1.0) <= c->refused_beta * 1.2) return FD_OK;
        fresh = true;
        FD_CUDA(c, cudaMemsetAsync(small, 0, 4, c->stream));
        k_far_pairs<<<128, 256, 0, c->stream>>>(c->xs(), L.DP, N, limit2, small);
        FD_LAUNCH_CHECK(c, "k_far_pairs");
        unsigned int far = 0;
        FD_CUDA(c, cudaMemcpyAsync(&far, small, 4, cudaMemcpyDeviceToHost, c->stream));
        FD_CUDA(c, cudaStreamSynchronize(c->stream));
        if ((double)far < 0.15 * 1024.0 * 1024.0) return FD_OK;
        // scratch: the operand buffers (re-packed in the new order afterwards); at least 64 bytes per point each
        int depth = 0;
        while (((int64_t)128 << depth) < N && depth < 12) ++depth;
        const int leaves = 1 << depth, blocks = (int)ceil_div(N, 1024);
        unsigned int* counts = c->at<unsigned int>(L.xp_col);
        char* scratch = c->at<char>(L.xp_row);
        unsigned short* leaf = reinterpret_cast<unsigned short*>(scratch);
        int* idx = reinterpret_cast<int*>(scratch + round_up(2 * N, 256));
        Node* nodes = reinterpret_cast<Node*>(idx + kSamples);
        unsigned int* totals = reinterpret_cast<unsigned int*>(nodes + kSamples);
        unsigned int* base = totals + kSamples;
        if (project) {
            // (scratch: counts are not needed yet)
            const double* mu = c->at<double>(L.mu);
            double* part = c->at<double>(L.part);
            const int n2 = L.DP * L.DP;
            k_cov_partial<<<kSamples / 128, 256, 128 * L.DP * 4, c->stream>>>(c->xs(), L.DP, N, mu, part);
            FD_LAUNCH_CHECK(c, "k_cov_partial");
            double* cov = part + (size_t)(kSamples / 128) * n2;
            k_cov_sum<<<(unsigned)ceil_div(n2, 256), 256, 0, c->stream>>>(part, kSamples / 128, n2, cov);
            FD_LAUNCH_CHECK(c, "k_cov_sum");
            std::vector<double> C((size_t)n2), lam, U;
            FD_CUDA(c, cudaMemcpyAsync(C.data(), cov, sizeof(double) * (size_t)n2, cudaMemcpyDeviceToHost, c->stream));
            FD_CUDA(c, cudaStreamSynchronize(c->stream));
            if (!sym_eig(C.data(), L.DP, lam, U)) { c->order_state = -1; return FD_OK; }
            Directions dir{};
            for (int d = 0; d < 8; ++d)
                for (int k = 0; k < L.DP; ++k) dir.v[d][k] = (float)U[k + (size_t)(L.DP - 1 - d) * L.DP];
            k_project<<<(unsigned)ceil_div(N, 256), 256, 0, c->stream>>>(c->xs(), L.DP, N, mu, dir, c->at<float>(L.zproj));
            FD_LAUNCH_CHECK(c, "k_project");
        }
        for (int l = 0; l < depth; ++l) {
            k_kd_level<<<1 << l, 512, 0, c->stream>>>(z, ZP, N, l, idx, nodes);
            FD_LAUNCH_CHECK(c, "k_kd_level");
        }
        k_kd_route<<<blocks, 1024, 0, c->stream>>>(z, ZP, N, depth, nodes, leaf, counts);
        FD_LAUNCH_CHECK(c, "k_kd_route");
        k_leaf_scan<<<(unsigned)ceil_div(leaves, 8), 256, 0, c->stream>>>(counts, blocks, leaves, totals);
        FD_LAUNCH_CHECK(c, "k_leaf_scan");
        k_scan<<<1, 1024, 0, c->stream>>>(totals, leaves, base);
        FD_LAUNCH_CHECK(c, "k_scan");
        k_scatter<<<blocks, 1024, 0, c->stream>>>(leaf, N, counts, base, leaves, perm);
        FD_LAUNCH_CHECK(c, "k_scatter");
        k_boxes<<<tiles, 128, 0, c->stream>>>(z, ZP, N, perm, box);
        FD_LAUNCH_CHECK(c, "k_boxes");
        c->order_state = 1;
        c->packed_beta = c->packed_row_beta = -1.0;
    }
    unsigned int* cnt = c->at<unsigned int>(L.list_counts);
    k_lists<<<pairs, 256, 0, c->stream>>>(box, ZP, tiles, limit2, c->at<unsigned short>(L.lists), cnt, cnt + pairs);
    FD_LAUNCH_CHECK(c, "k_lists");
    unsigned int* offs = cnt + 2 * pairs;
    k_scan<<<1, 1024, 0, c->stream>>>(cnt, pairs, offs);
    FD_LAUNCH_CHECK(c, "k_scan");
    k_scan<<<1, 1024, 0, c->stream>>>(cnt + pairs, pairs, offs + pairs + 1);
    FD_LAUNCH_CHECK(c, "k_scan");
    c->listed_kind = kind; c->listed_beta = beta;
    if (known) return FD_OK;
    unsigned int total = 0;
    FD_CUDA(c, cudaMemcpyAsync(&total, offs + pairs, 4, cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    st.total = total;
    st.on = (double)total < 0.9 * (double)pairs * (double)tiles;
    if (fresh && !st.on) {
        // nothing gained: the points keep the caller's order (a larger bandwidth may try again)
        c->order_state = 0;
        c->refused_beta = std::max(c->refused_beta, beta * (kind == 0 ? 60.25 / 40.25 : 1.0));
    }
    return FD_OK;
}

}  // namespace fd
