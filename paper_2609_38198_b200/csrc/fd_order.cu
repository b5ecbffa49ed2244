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
// Order: a k-d tree over up to 4096 sampled points (each node splits its samples at the median of their widest coordinate) down to
// leaves of about 128 points (16 where the direct-difference kernels may use it); all points are routed through it and sorted by
// leaf, stably.  It is made once per context, by the degree passes of a bandwidth with many pairs beyond the exponent limit; the
// degree passes of a new context then take 0.1 (N = 16384, D = 4) to 0.6 ms (N = 2^18, D = 30) longer, which one of the
// two passes or the first products pay back from 16384 points on in the plane and on surfaces (direct differences; N = 8192: 130 us of
// passes against 300) and from 32768 on in the Gram form.  Vectors stay in the caller's order everywhere: packing and staging
// gather through the permutation, the epilogues scatter.  Gram-form passes at a bandwidth with lists work in the order, all others (and
// direct-difference passes without lists) in the caller's.
//
// Lists by the boxes: for a bandwidth and exponent limit, per 256 rows the column tiles of 128 points whose bounding box comes close enough
// (distance of the two boxes: a lower bound for every pair); for the direct-difference kernels per 64 rows the tiles of 16 points, there
// against the 4 boxes of the rows, too.  Data that fill many dimensions (the 6-torus) have no far tiles; then the passes run over all
// tiles as before.
//
// Lists by notes: boxes of curved patches leave a third more tiles than hold a near pair.  The first degree pass computes every kernel value
// anyway, so it notes which tiles had one within the limits (from the sums of squares that it forms anyway; direct differences: from the
// sums), and the second pass and the products at that bandwidth go by these notes.  R^30 on a two-dimensional manifold, beta = 2: 0.80 -> 0.64 of the
// tiles at N = 65536 (b = 32: 1225 -> 975 us a product), 0.67 -> 0.58 at N = 2^18 (20.0 -> 17.3 ms); 2-torus, direct differences: 0.26 -> 0.17 at
// N = 16384, beta = 100, 0.56 -> 0.39 at N = 65536, beta = 30.  The first pass goes by the boxes always, so that its results do not depend on earlier calls.
//
// (The extension's new points in an order of their own, listed by the boxes: 40009 points against 65536 leave 0.88 of the tiles, and what
// that saves goes into the order: 985 -> 965 us; 16500 against 33000: 290 -> 319.  They are taken as they come.)
#include <algorithm>
#include <cmath>
#include <new>

#include "fd_dense.h"

namespace fd {

namespace {

constexpr int kSamples = 4096;

// Counts pairs of 512 sampled points farther apart than limit2 (squared distance), and those within a quarter of that distance.
__global__ void __launch_bounds__(256)
k_far_pairs(const float* __restrict__ xs, int DP, int64_t n, float limit2, unsigned int* __restrict__ count) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;      // one sampled row per warp
    const float* xi = xs + (n * i / 512) * DP;
    unsigned int far = 0, close = 0;
    for (int j = lane; j < 512; j += 32) {
        const float* xj = xs + (n * j / 512) * DP;
        float d2 = 0.f;
        for (int k = 0; k < DP; ++k) { const float d = xi[k] - xj[k]; d2 = fmaf(d, d, d2); }
        far += d2 > limit2;
        close += d2 <= 0.0625f * limit2;
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) { far += __shfl_xor_sync(0xffffffffu, far, m); close += __shfl_xor_sync(0xffffffffu, close, m); }
    if (lane == 0) { atomicAdd(count, far); atomicAdd(count + 1, close); }
}

// Whether lists by the boxes are expected to leave out enough, from the sampled pairs: `far` of 512 x 512 beyond the limit, `close` within a quarter
// of its distance r.  The two counts give the data's dimension d at that scale (near pairs within a distance grow with its d-th power), this
// the radius of the tiles, and tiles count as near up to r and their two radii (twice these where tiles are of 128 points and boxes larger).
// 19 data sets (circles, tori, spheres, boxes, normal clouds, clusters and lines in 2 to 8 coordinates), N = 16384 .. 32000: direct differences:
// lists that were used were predicted at up to 0.75 of the tiles, those refused from 0.76 on (two: 0.67, 0.68); Gram form up to 1.00 and, most of
// them, from 1.05 on (eight: 0.88 to 0.99).
bool lists_expected(unsigned int far, unsigned int close, int64_t N, bool direct) {
    constexpr double kPairs = 512.0 * 512.0;
    const double near = std::max(1.0 - far / kPairs - 1.0 / 512.0, 1.0 / kPairs), mid = std::max((double)close - 512.0, 1.0) / kPairs;   // (without the points themselves)
    const double d = std::max(std::log(near / mid) / std::log(4.0), 0.05);
    auto radius = [&](double points) { return std::pow(points / ((double)N * near), 1.0 / d); };
    const double reach = direct ? radius(64.0) + radius(16.0) : 2.0 * (radius(256.0) + radius(128.0));
    return near * std::pow(1.0 + reach, d) < (direct ? 0.77 : 1.04);
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

// The tree over S = 1024 E evenly spaced points: nodes of level l at nodes[2^l - 1 ..].  One CTA with the samples' coordinates (at most 8) in
// shared memory; a level is the extent of every node's samples, then one bitonic sort of all nodes' segments at once.  A thread holds
// entries warp * 32 E + 32 u + lane: exchanges closer than 32 E go through shuffles and registers (S = 2048: 250 of 285; all through
// shared memory took 146 us, a launch per level 120 us).
constexpr int kKdThr = 1024;
constexpr int kd_smem(int samples, int DP) { return samples * (DP * 4 + 8) + (samples / 32) * 16 * 4 + (samples / 2) * 4; }
template <int E>
__global__ void __launch_bounds__(kKdThr)
k_kd_tree(const float* __restrict__ xs, int DP, int64_t n, int depth, Node* __restrict__ nodes) {
    constexpr int S = kKdThr * E;
    extern __shared__ __align__(16) float kd[];
    float* coord = kd;                                             // [DP][S]
    float* skey = coord + (size_t)S * DP;
    int* sval = reinterpret_cast<int*>(skey + S);
    float (*chunk)[2][8] = reinterpret_cast<float(*)[2][8]>(sval + S);             // extents of 32 consecutive entries
    int* dim = reinterpret_cast<int*>(chunk + S / 32);                             // of each node
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e0 = warp * 32 * E + lane;
    for (int t = threadIdx.x; t < S; t += kKdThr) {
        const float* x = xs + (n * t / S) * DP;
        for (int k = 0; k < DP; ++k) coord[k * S + t] = x[k];
    }
    float key[E];
    int val[E];
#pragma unroll
    for (int u = 0; u < E; ++u) val[u] = e0 + 32 * u;
    __syncthreads();
    for (int level = 0; level < depth; ++level) {
        const int len = S >> level;
        // widest coordinate of every node
        const int width = len < 32 ? len : 32;
#pragma unroll
        for (int u = 0; u < E; ++u) {
            float widest = -1.f;
            int d = 0;
            for (int k = 0; k < DP; ++k) {
                float lo = coord[k * S + val[u]], hi = lo;
                for (int m = width >> 1; m >= 1; m >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m)); }
                if (hi - lo > widest) { widest = hi - lo; d = k; }
                if (len >= 32 && lane == 0) { chunk[warp * E + u][0][k] = lo; chunk[warp * E + u][1][k] = hi; }
            }
            const int e = e0 + 32 * u;
            if (len < 32 && e % len == 0) dim[e / len] = d;
        }
        __syncthreads();
        if (len >= 32) {
            const int per = len / 32;                              // chunks of a node; a warp per node
            for (int node = warp; node < (1 << level); node += kKdThr / 32) {
                float widest = -1.f;
                int d = 0;
                for (int k = 0; k < DP; ++k) {
                    float lo = INFINITY, hi = -INFINITY;
                    for (int q = lane; q < per; q += 32) { lo = fminf(lo, chunk[node * per + q][0][k]); hi = fmaxf(hi, chunk[node * per + q][1][k]); }
#pragma unroll
                    for (int m = 16; m >= 1; m >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m)); }
                    if (hi - lo > widest) { widest = hi - lo; d = k; }
                }
                if (lane == 0) dim[node] = d;
            }
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < E; ++u) key[u] = coord[dim[(e0 + 32 * u) / len] * S + val[u]];
        for (int size = 2; size <= len; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                float ok[E];
                int ov[E];
                if (stride >= 32 * E) {
#pragma unroll
                    for (int u = 0; u < E; ++u) { skey[e0 + 32 * u] = key[u]; sval[e0 + 32 * u] = val[u]; }
                    __syncthreads();
#pragma unroll
                    for (int u = 0; u < E; ++u) { ok[u] = skey[(e0 + 32 * u) ^ stride]; ov[u] = sval[(e0 + 32 * u) ^ stride]; }
                    __syncthreads();
                } else if (stride >= 32) {
#pragma unroll
                    for (int u = 0; u < E; ++u) {
                        ok[u] = stride == 32 ? key[(u ^ 1) % E] : key[(u ^ 2) % E];
                        ov[u] = stride == 32 ? val[(u ^ 1) % E] : val[(u ^ 2) % E];
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < E; ++u) { ok[u] = __shfl_xor_sync(0xffffffffu, key[u], stride); ov[u] = __shfl_xor_sync(0xffffffffu, val[u], stride); }
                }
#pragma unroll
                for (int u = 0; u < E; ++u) {
                    const int e = e0 + 32 * u;
                    const bool up = size == len || (e & size) == 0, lower = (e & stride) == 0;
                    const bool gt = key[u] > ok[u] || (key[u] == ok[u] && val[u] > ov[u]);     // ties by index: the order is unique
                    if ((lower == up) == gt) { key[u] = ok[u]; val[u] = ov[u]; }
                }
            }
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int e = e0 + 32 * u;
            if (e % len == len / 2) nodes[(1 << level) - 1 + e / len] = Node{dim[e / len], key[u]};
        }
        __syncthreads();
    }
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

// The points in their order, padded with points whose squared distance from any other overflows (kernel value 0: lists are used only where
// |x|^2 beta is a normal number).  Points 1e18 away are among those of a data set of that scale, and row sums count what they see.
__global__ void __launch_bounds__(256)
k_order_points(const float4* __restrict__ xs, int DP4, int64_t n, int64_t np, const int* __restrict__ perm, float4* __restrict__ out) {
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= np) return;
    const int64_t i = p < n ? perm[p] : -1;
    for (int k = 0; k < DP4; ++k) out[p * DP4 + k] = i >= 0 ? xs[i * DP4 + k] : make_float4(3e38f, 3e38f, 3e38f, 3e38f);
}

// Bounding box of each tile of 16 consecutive positions, for up to 8 coordinates: 16 lanes a tile.
__global__ void __launch_bounds__(256)
k_boxes16(const float* __restrict__ xs, int DP, int64_t n, const int* __restrict__ perm, int tiles, float* __restrict__ box) {
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t i = p < n ? perm[p] : -1;
    for (int k = 0; k < DP; ++k) {
        float lo = INFINITY, hi = -INFINITY;
        if (i >= 0) lo = hi = xs[i * DP + k];
#pragma unroll
        for (int m = 8; m >= 1; m >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m)); }
        if ((threadIdx.x & 15) == 0 && p / 16 < tiles) {
            box[(size_t)(p / 16) * 2 * DP + k] = lo;
            box[((size_t)(p / 16) * 2 + 1) * DP + k] = hi;
        }
    }
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

// Column tiles (per_pair to a row pair) of row pair blockIdx.x whose box comes within limit2 of the pair's box, ascending: list[pair * tiles ..];
// counts[pair] of them, of which `upper[pair]` are the pair's own and later ones (the symmetric row sums start there).
// noted (null: by the boxes): what a row-sum pass saw, note_rows rows of `tiles` entries for a pair, not 0 for near ones.
__global__ void __launch_bounds__(1024)
k_lists(const float* __restrict__ box, int DP, int tiles, int per_pair, float limit2, const unsigned char* __restrict__ noted, int note_rows,
        unsigned short* __restrict__ list, unsigned int* __restrict__ counts, unsigned int* __restrict__ upper) {
    __shared__ float lo[64], hi[64];
    __shared__ float sub[4][2][8];                                     // boxes of the row tiles (per_pair = 4, up to 8 coordinates)
    __shared__ unsigned int wsum[32];
    const int pair = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < DP && !noted; k += 1024) {
        float l = INFINITY, h = -INFINITY;
        for (int t = 0; t < per_pair; ++t) {
            const float* a = box + ((size_t)pair * per_pair + t) * 2 * DP;
            l = fminf(l, a[k]); h = fmaxf(h, a[DP + k]);
            if (per_pair == 4) { sub[t][0][k] = a[k]; sub[t][1][k] = a[DP + k]; }
        }
        lo[k] = l; hi[k] = h;
    }
    __syncthreads();
    unsigned int n = 0, below = 0;
    for (int t0 = 0; t0 < tiles; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        bool near = false;
        if (t < tiles && noted) {
            for (int s = 0; s < note_rows; ++s) near = near || noted[((size_t)pair * note_rows + s) * tiles + t] != 0;
            near = near || t / per_pair == pair;
        } else if (t < tiles) {
            const float* b = box + (size_t)t * 2 * DP;
            float d2 = 0.f;
            for (int k = 0; k < DP; ++k) {
                const float g = fmaxf(fmaxf(b[k] - hi[k], lo[k] - b[DP + k]), 0.f);
                d2 = fmaf(g, g, d2);
            }
            near = d2 <= limit2;
            if (near && per_pair == 4) {
                // near the box of all 64 rows: near one of the 4 smaller boxes?
                near = false;
                for (int s = 0; s < 4 && !near; ++s) {
                    float e2 = 0.f;
                    for (int k = 0; k < DP; ++k) {
                        const float g = fmaxf(fmaxf(b[k] - sub[s][1][k], sub[s][0][k] - b[DP + k]), 0.f);
                        e2 = fmaf(g, g, e2);
                    }
                    near = e2 <= limit2;
                }
            }
            near = near || t / per_pair == pair;                   // (an empty box is infinitely far; a pair's own tiles always count)
        }
        const unsigned int vote = __ballot_sync(0xffffffffu, near);
        if (lane == 0) wsum[warp] = __popc(vote);
        __syncthreads();
        unsigned int pos = n + __popc(vote & ((1u << lane) - 1u)), all = 0;
        for (int w = 0; w < 32; ++w) { if (w < warp) pos += wsum[w]; all += wsum[w]; }
        if (near) {
            list[(size_t)pair * tiles + pos] = (unsigned short)t;
            if (t == per_pair * pair) below = pos + 1;                        // (one thread of the block sees it)
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
    auto& st = c->lists[kind == 3 ? 1 : kind == 4 ? 2 : kind];
    if (L.perm == 0 || c->order_state < 0) return FD_OK;
    const bool direct = kind == 2 || kind == 4;
    const bool noted = c->near_beta == beta && c->near_direct == direct && kind != 1 && kind != 2;
    if (kind == 3 && L.near == 0) kind = 1;                        // (one buffer for all, by the boxes: the first degree pass's lists serve the second)
    const int buf = L.near == 0 || kind == 0 || kind == 4 ? 0 : kind == 3 ? 2 : 1;
    auto& listed = c->listed[buf];
    const int held = noted ? 8 + kind : kind;                      // what the buffer would hold
    if (st.beta == beta && (!st.on || (!c->captured && listed.kind == held && listed.beta == beta))) return FD_OK;
    // Beyond an exponent of 40 both fp16 pieces of a kernel value are zero (2^15 2^-40 = 2^-25 rounds to zero), beyond 60 a degree
    // contribution is below the fixed-point unit; the quarter covers the rounding of the boxes' distance.
    // The direct-difference kernels' exponential gives exactly zero beyond 126.
    const double limit = kind == 0 ? 40.25 : direct ? 126.25 : 60.25;
    const double scaled_beta = beta * (60.25 / limit);             // bandwidths of the kinds on one scale
    if (direct && !L.direct_lists) return FD_OK;
    if (!decide && st.beta != beta) return FD_OK;
    const bool known = st.beta == beta;                            // decided before, only overwritten by the other kind's lists
    const int64_t N = L.N;
    // rows of a list, tiles of a row of tiles
    const int per_pair = direct ? 4 : 2, pairs = (int)(L.NP / (direct ? 64 : 256)), tiles = pairs * per_pair;
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
        if (scaled_beta <= c->refused_beta * 1.2) return FD_OK;
        fresh = true;
        FD_CUDA(c, cudaMemsetAsync(small, 0, 8, c->stream));
        k_far_pairs<<<64, 256, 0, c->stream>>>(c->xs(), L.DP, N, limit2, small);
        FD_LAUNCH_CHECK(c, "k_far_pairs");
        unsigned int count[2] = {0, 0};
        FD_CUDA(c, cudaMemcpyAsync(count, small, 8, cudaMemcpyDeviceToHost, c->stream));
        FD_CUDA(c, cudaStreamSynchronize(c->stream));
        // Share of far pairs from which an order is tried: 0.4.  Below 32768 points it costs as much as the pass itself (190 to 450 us), so that between
        // 0.4 and 0.8 it is made only where it is expected to stay: first degree pass, N = 20000: 6-dimensional data 1120 -> 720 us, 2-torus at
        // beta = 20 834 -> 520.  Where it stays, two to five products at the bandwidth pay for it (2-torus, N = 16384, beta = 30: 100 us for 153
        // a product of 16 columns; circle, Gram form, beta = 20: 177 us for 36).
        if ((double)count[0] < 0.4 * 512.0 * 512.0) return FD_OK;
        if (N < 32768 && (double)count[0] < 0.8 * 512.0 * 512.0 && !lists_expected(count[0], count[1], N, direct)) return FD_OK;
        // scratch: the operand buffers (re-packed in the new order afterwards); at least 64 bytes per point each
        int depth = 0;
        while (((int64_t)(L.direct_lists ? 16 : 128) << depth) < N && depth < 12) ++depth;
        const int samples = std::min(kSamples, std::max(1024, 2 << depth));        // two to a leaf or more, where there are as many
        const int leaves = 1 << depth, blocks = (int)ceil_div(N, 1024);
        unsigned int* counts = c->at<unsigned int>(L.xp_col);
        char* scratch = c->at<char>(L.xp_row);
        unsigned short* leaf = reinterpret_cast<unsigned short*>(scratch);
        Node* nodes = reinterpret_cast<Node*>(scratch + round_up(2 * N, 256));
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
            double C[64 * 64];
            FD_CUDA(c, cudaMemcpyAsync(C, cov, sizeof(double) * (size_t)n2, cudaMemcpyDeviceToHost, c->stream));
            FD_CUDA(c, cudaStreamSynchronize(c->stream));
            Directions dir{};
            bool solved = false;
            try {
                std::vector<double> lam, U;
                solved = sym_eig(C, L.DP, lam, U);
                for (int d = 0; d < 8 && solved; ++d)
                    for (int k = 0; k < L.DP; ++k) dir.v[d][k] = (float)U[k + (size_t)(L.DP - 1 - d) * L.DP];
            } catch (const std::bad_alloc&) {}                     // (nothing may be thrown through the C interface)
            if (!solved) { c->order_state = -1; return FD_OK; }
            k_project<<<(unsigned)ceil_div(N, 256), 256, 0, c->stream>>>(c->xs(), L.DP, N, mu, dir, c->at<float>(L.zproj));
            FD_LAUNCH_CHECK(c, "k_project");
        }
        const int smem = kd_smem(samples, ZP);
        const auto tree = samples == 1024 ? k_kd_tree<1> : samples == 2048 ? k_kd_tree<2> : k_kd_tree<4>;
        FD_CUDA(c, cudaFuncSetAttribute(tree, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        tree<<<1, kKdThr, smem, c->stream>>>(z, ZP, N, depth, nodes);
        FD_LAUNCH_CHECK(c, "k_kd_tree");
        k_kd_route<<<blocks, 1024, 0, c->stream>>>(z, ZP, N, depth, nodes, leaf, counts);
        FD_LAUNCH_CHECK(c, "k_kd_route");
        k_leaf_scan<<<(unsigned)ceil_div(leaves, 8), 256, 0, c->stream>>>(counts, blocks, leaves, totals);
        FD_LAUNCH_CHECK(c, "k_leaf_scan");
        k_scan<<<1, 1024, 0, c->stream>>>(totals, leaves, base);
        FD_LAUNCH_CHECK(c, "k_scan");
        k_scatter<<<blocks, 1024, 0, c->stream>>>(leaf, N, counts, base, leaves, perm);
        FD_LAUNCH_CHECK(c, "k_scatter");
        if (L.direct_lists) {
            k_order_points<<<(unsigned)ceil_div(L.NP, 256), 256, 0, c->stream>>>(reinterpret_cast<const float4*>(c->xs()), L.DP / 4, N, L.NP, perm, c->at<float4>(L.xord));
            FD_LAUNCH_CHECK(c, "k_order_points");
        }
        c->order_state = 1;
        c->boxes_kind = -1;
        c->packed_beta = c->packed_row_beta = -1.0;
    }
    if (c->captured || c->boxes_kind != (direct ? 1 : 0)) {
        if (direct) k_boxes16<<<(unsigned)ceil_div(L.NP, 256), 256, 0, c->stream>>>(z, ZP, N, perm, tiles, box);
        else k_boxes<<<tiles, 128, 0, c->stream>>>(z, ZP, N, perm, box);
        FD_LAUNCH_CHECK(c, "k_boxes");
        c->boxes_kind = direct ? 1 : 0;
    }
    unsigned int* cnt = c->at<unsigned int>(L.list_counts[buf]);
    const unsigned char* notes = noted ? c->at<unsigned char>(L.near) + (kind == 3 ? (size_t)tiles * tiles : 0) : nullptr;
    k_lists<<<pairs, 1024, 0, c->stream>>>(box, ZP, tiles, per_pair, limit2, notes, direct ? 1 : 2, c->at<unsigned short>(L.lists[buf]), cnt, cnt + pairs);
    FD_LAUNCH_CHECK(c, "k_lists");
    unsigned int* offs = cnt + 2 * pairs;
    // offsets of all entries, and of the upper ones (degree passes in the Gram form)
    if (kind != 3) {
        k_scan<<<1, 1024, 0, c->stream>>>(cnt, pairs, offs);
        FD_LAUNCH_CHECK(c, "k_scan");
    }
    if (kind == 1 || kind == 3) {
        k_scan<<<1, 1024, 0, c->stream>>>(cnt + pairs, pairs, offs + pairs + 1);
        FD_LAUNCH_CHECK(c, "k_scan");
    }
    listed.kind = held; listed.beta = beta;
    if (known) return FD_OK;
    unsigned int total = 0;
    FD_CUDA(c, cudaMemcpyAsync(&total, offs + pairs, 4, cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    st.total = total;
    st.on = (double)total < (direct ? 0.8 : 0.9) * (double)pairs * (double)tiles;
    if (fresh && !st.on) {
        // nothing gained: the points keep the caller's order (a larger bandwidth may try again)
        c->order_state = 0;
        c->refused_beta = std::max(c->refused_beta, scaled_beta);
    }
    return FD_OK;
}

}  // namespace fd
