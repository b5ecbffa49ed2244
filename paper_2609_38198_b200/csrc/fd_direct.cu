// Direct-difference fp32 kernels on the FMA pipe (Eqs. 5-6 with the distance taken as
// sum_k (x_ik - x_jk)^2 instead of the Gram form of Eq. 4).
//
// This family serves the shapes where the Gram form is not accurate enough in fp32 (small D
// with large beta * |x|^2: the circle and 2-torus workloads) and every shape the tensor-core
// kernels do not cover.
//
// A work step is a tile of 256 rows x 64 (small problems: 16) columns (points j).  The flat sequence of (row tile, column tile) steps is cut into equal ranges,
// one per resident CTA (two to four per SM), so any size fills the GPU evenly.  A row tile that a cut falls into is finished by
// k_direct_fix: every CTA leaves its share in a slot of its own and the shares are added in the order of the CTAs, so
// results are bit-reproducible run to run.  (Letting the CTA that comes last add them needs no second launch but puts one
// CTA's chain of dependent reads at the end: 183 us instead of 8 at N = 2048.)
//
// What bounds it: instruction issue and the latency between dependent instructions, 2 D + b + 2 FMA-pipe operations per pair (N = 12000,
// D = 4, b = 16: 74 % of the issue slots taken, FMA pipe 62 %, 2.0 eligible warps a scheduler).  A thread owns two or four rows (four: the two halves of the
// CTA take half the columns of a tile each), which share the broadcast reads of x_j and w_j from shared memory; with one row per
// thread these cost as many slots as a fifth of the FMAs.  (Two rows per packed instruction, add / fma.rn.f32x2, halve
// the instruction count but ran at half the FMA rate: 5 to 15 % slower in every shape; two columns per packed instruction gain for 64 columns, fd_direct.h.)  Right-hand columns are read from V
// as it is (column-major) and scaled on the way into shared memory: no packing pass.
// N = 16384, D = 4, b = 16: 412 -> 309 us a product; N = 12000, D = 12, b = 48: 944 -> 639 us; N = 6000, D = 2, both degree passes:
// 136 -> 109 us (one row per thread, separate packing pass, one CTA more or less per SM at the end).
//
// Up to 8 coordinates, from 16384 points on, passes over the whole point set may run over tile lists instead: fd_direct_listed.cu.
#include <cooperative_groups.h>

#include <algorithm>

#include "fd_direct.h"

namespace fd {

namespace {

using namespace direct;

constexpr int kRowsT = 256;      // rows per row tile
constexpr int kTJ = 64;          // points per column tile, at most (DirectParams::tj_log2)
constexpr int kFlushCols = 2048; // columns between flushes of the fp32 tile accumulators
constexpr int kMaxCtasPerSm = 4; // (the shares of cut row tiles are provisioned for four)

struct DirectParams {
    const float4* xrow; const float4* xcol;      // padded points, DP4 float4 each
    int64_t Nrow, N;
    float nbeta2;                                // -beta log2(e)
    const float* V; int64_t ldv; int vcols;      // block mode: right block, columns from vcols on are the ones vector
    const float* right; const float* left;       // may be null
    float* Y; int64_t ldy; int b;
    double* rowsq;                               // row-sum mode: sum_j K_ij^2 (may be null); Y = the weighted row sums
    void* part;                                  // 2 slots per CTA: shares of row tiles that are cut
    int row_tiles, col_tiles;
    int tj_log2;                                 // log2 of the points per column tile: 6, or 4 where 64 would leave too few steps
};

__host__ __device__ __forceinline__ long long range_begin(long long total, int cta, int ctas) { return total * cta / ctas; }
// (A CTA's share of a row tile goes to its slot 1 if its range holds the row tile's first step, else to slot 0.)

// A CTA's range of steps, one row tile after the other.
struct Range {
    long long g, g_end;
    int rt = -1, c0, n;                              // steps c0 .. c0 + n of the row tile
    __device__ __forceinline__ Range(const DirectParams& p) {
        const long long total = (long long)p.row_tiles * p.col_tiles;
        g = range_begin(total, (int)blockIdx.x, (int)gridDim.x);
        g_end = range_begin(total, (int)blockIdx.x + 1, (int)gridDim.x);
    }
    __device__ __forceinline__ bool next(const DirectParams& p) {
        if (g >= g_end) return false;                // (the same for the whole CTA)
        rt = (int)(g / p.col_tiles);
        c0 = (int)(g - (long long)rt * p.col_tiles);
        n = (int)(p.col_tiles - c0 < g_end - g ? p.col_tiles - c0 : g_end - g);
        g += n;
        return true;
    }
};

// Stages the points of a column tile (padding points lie 1e18 away: kernel value 0).
template <int DP4>
__device__ __forceinline__ void stage_points(const DirectParams& p, int64_t j0, float4* sx) {
    for (int t = threadIdx.x; t < (DP4 << p.tj_log2); t += kThr) {
        const int64_t j = j0 + t / DP4;
        sx[t] = j < p.N ? p.xcol[j0 * DP4 + t] : make_float4(1e18f, 1e18f, 1e18f, 1e18f);
    }
}

// Row r of a thread: position lane_row + (256 / R) r of the row tile.
template <int DP4, int R>
__device__ __forceinline__ void load_rows(const DirectParams& p, int64_t row0, int lane_row, float4 (&xi)[R][DP4]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = row0 + lane_row + (kRowsT / R) * r;
        const bool valid = i < p.Nrow;
#pragma unroll
        for (int k = 0; k < DP4; ++k) xi[r][k] = valid ? p.xrow[i * DP4 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

template <bool COPY, int R, int BT, class S>
__device__ __forceinline__ float (&after_loop(float (&copy)[R][BT], S& acc))[R][BT] {
    if constexpr (COPY) return copy;
    else return acc.v;
}

// Block mode: Y[i, c] = left_i sum_j K_ij right_j V[j, c] for c < b <= BT.
// (resident CTAs asked for: four, three or two, by the registers that the rows and sums of a thread need)
constexpr int min_ctas(int regs) { return regs + 40 <= 128 ? 4 : regs + 40 <= 168 ? 3 : 2; }
template <int DP4, int BT, int R>
__global__ void __launch_bounds__(kThr, min_ctas(R * (4 * DP4 + BT)))
k_direct(const DirectParams p) {
    constexpr int H = R * kThr / kRowsT;               // column parts of a tile (R = 4: 2)
    constexpr int BP = BT + 4;                         // pitch of the staged block (16-byte rows; spreads the transposing stores)
    extern __shared__ __align__(16) float smem[];
    float4* sx = reinterpret_cast<float4*>(smem);                       // kTJ x DP4
    float* sw = smem + kTJ * DP4 * 4;                                   // kTJ x BP
    float* sacc = sw + kTJ * BP;                                        // [H][BT][256]: flushed sums
    const int part = H == 1 ? 0 : (int)threadIdx.x / (kThr / H);
    const int lane_row = H == 1 ? (int)threadIdx.x : (int)threadIdx.x % (kThr / H);
    const int tj = 1 << p.tj_log2;
    for (Range range(p); range.next(p);) {
        const int c0 = range.c0, n = range.n;
        const int64_t row0 = (int64_t)range.rt * kRowsT;
        float4 xi[R][DP4];
        load_rows<DP4, R>(p, row0, lane_row, xi);
        Sums<R, BT, (BT > 48 && DP4 != 5 && DP4 != 6)> acc;              // (packed, 17 to 24 coordinates spill 72 and 236 bytes a thread)
        // After the loop the sums are worked on where they are, or in a copy: where the loop's are packed, and where the compiler spills less with a
        // copy (up to 4 coordinates, 32 columns: 0 instead of 44 bytes a thread, 1 to 3 % faster; up to 12, 48: 44 instead of 68, 4 %).  In the
        // other shapes a copy, or add() instead of the plain loop below, costs up to 7 % (N = 12000, b = 12 and 16: D = 4 179 and 181 instead of
        // 166 and 171 us, D = 12 267 and 274 instead of 262 and 270; b = 8, D = 4: 120 instead of 115).
        constexpr bool kCopy = (BT > 48 && DP4 != 5 && DP4 != 6) || (DP4 == 1 && BT == 32) || (DP4 == 3 && BT == 48);
        float copy[R][BT];
        acc.clear();
        // a thread's own slots of sacc: row r, column c at mine[c * 256 + (256 / R) * r]
        float* mine = sacc + part * BT * kRowsT + lane_row;
        bool flushed = false;
        for (int t = 0; t < n; ++t) {
            const int64_t j0 = (int64_t)(c0 + t) << p.tj_log2;
            __syncthreads();
            stage_points<DP4>(p, j0, sx);
            for (int e = threadIdx.x; e < (BT << p.tj_log2); e += kThr) {
                const int jj = e & (tj - 1), c = e >> p.tj_log2;   // rows of V fastest: coalesced
                const int64_t j = j0 + jj;
                float w = 0.f;
                if (c < p.b && j < p.N) {
                    w = c < p.vcols ? p.V[j + (int64_t)c * p.ldv] : 1.f;
                    if (p.right) w *= p.right[j];
                }
                sw[jj * BP + c] = w;
            }
            __syncthreads();
#pragma unroll 2
            for (int jj = part * (tj / H); jj < (part + 1) * (tj / H); ++jj) {
                float kij[R];
                kernel_values<DP4, R>(sx, jj, xi, p.nbeta2, kij);
                if constexpr (kCopy) acc.add(kij, reinterpret_cast<const float4*>(&sw[jj * BP]));
                else {
#pragma unroll
                    for (int c4 = 0; c4 < BT / 4; ++c4) {
                        const float4 w = *reinterpret_cast<const float4*>(&sw[jj * BP + 4 * c4]);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            acc.v[r][4 * c4 + 0] = fmaf(kij[r], w.x, acc.v[r][4 * c4 + 0]);
                            acc.v[r][4 * c4 + 1] = fmaf(kij[r], w.y, acc.v[r][4 * c4 + 1]);
                            acc.v[r][4 * c4 + 2] = fmaf(kij[r], w.z, acc.v[r][4 * c4 + 2]);
                            acc.v[r][4 * c4 + 3] = fmaf(kij[r], w.w, acc.v[r][4 * c4 + 3]);
                        }
                    }
                }
            }
            if (((t + 1) & (kFlushCols / tj - 1)) == 0 && t + 1 < n) {
                // two-level summation keeps the rounding error of long column ranges at the 1e-7 level
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < BT; ++c) {
                        float* s = mine + c * kRowsT + (kRowsT / R) * r;
                        *s = flushed ? *s + acc.get(r, c) : acc.get(r, c);
                    }
                acc.clear();
                flushed = true;
            }
        }
        if (kCopy) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < BT; ++c) copy[r][c] = acc.get(r, c);
        }
        float (&sum)[R][BT] = after_loop<kCopy>(copy, acc);
        if (flushed) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < BT; ++c) sum[r][c] += mine[c * kRowsT + (kRowsT / R) * r];
        }
        if (H == 2) {
            // the second half hands its sums to the first
            if (part == 1) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < BT; ++c) mine[c * kRowsT + (kRowsT / R) * r] = sum[r][c];
            }
            __syncthreads();
            if (part == 0) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < BT; ++c) sum[r][c] += mine[(BT + c) * kRowsT + (kRowsT / R) * r];
            }
        }
        if (part == 0) {
            const bool whole = n == p.col_tiles;
            float* slot = static_cast<float*>(p.part) +
                          (size_t)(2 * blockIdx.x + (c0 == 0 ? 1 : 0)) * BT * kRowsT + lane_row;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = row0 + lane_row + (kRowsT / R) * r;
                const bool valid = i < p.Nrow;
                const float l = whole && p.left && valid ? p.left[i] : 1.0f;
#pragma unroll
                for (int c = 0; c < BT; ++c)
                    if (c < p.b) {
                        if (!whole) slot[c * kRowsT + (kRowsT / R) * r] = sum[r][c];
                        else if (valid) p.Y[i + (int64_t)c * p.ldy] = sum[r][c] * l;
                    }
            }
        }
    }
    grid_go();
}

// Row-sum mode: sum_j K_ij right_j and sum_j K_ij^2; a column tile (<= 64 terms) in fp32, across tiles in fp64.
template <int DP4>
__global__ void __launch_bounds__(kThr)
k_direct_rowsum(const DirectParams p) {
    constexpr int R = DP4 <= 4 ? 4 : 2, H = R * kThr / kRowsT;
    __shared__ float4 sx[kTJ * DP4];
    __shared__ float sw[kTJ];
    __shared__ double2 sacc[kRowsT];
    const int part = H == 1 ? 0 : (int)threadIdx.x / (kThr / H);
    const int lane_row = H == 1 ? (int)threadIdx.x : (int)threadIdx.x % (kThr / H);
    const int tj = 1 << p.tj_log2;
    for (Range range(p); range.next(p);) {
        const int c0 = range.c0, n = range.n;
        const int64_t row0 = (int64_t)range.rt * kRowsT;
        float4 xi[R][DP4];
        load_rows<DP4, R>(p, row0, lane_row, xi);
        double dsum[R], dsq[R];
#pragma unroll
        for (int r = 0; r < R; ++r) { dsum[r] = 0.0; dsq[r] = 0.0; }
        for (int t = 0; t < n; ++t) {
            const int64_t j0 = (int64_t)(c0 + t) << p.tj_log2;
            __syncthreads();
            stage_points<DP4>(p, j0, sx);
            if ((int)threadIdx.x < tj) {
                const int64_t j = j0 + threadIdx.x;
                sw[threadIdx.x] = j < p.N ? (p.right ? p.right[j] : 1.0f) : 0.f;
            }
            __syncthreads();
            float a[R], q[R];
#pragma unroll
            for (int r = 0; r < R; ++r) { a[r] = 0.f; q[r] = 0.f; }
#pragma unroll 4
            for (int jj = part * (tj / H); jj < (part + 1) * (tj / H); ++jj) {
                float kij[R];
                kernel_values<DP4, R>(sx, jj, xi, p.nbeta2, kij);
                const float w = sw[jj];
#pragma unroll
                for (int r = 0; r < R; ++r) { a[r] = fmaf(kij[r], w, a[r]); q[r] = fmaf(kij[r], kij[r], q[r]); }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) { dsum[r] += (double)a[r]; dsq[r] += (double)q[r]; }
        }
        if (H == 2) {
            __syncthreads();
            if (part == 1) {
#pragma unroll
                for (int r = 0; r < R; ++r) sacc[lane_row + (kRowsT / R) * r] = make_double2(dsum[r], dsq[r]);
            }
            __syncthreads();
            if (part == 0) {
#pragma unroll
                for (int r = 0; r < R; ++r) { const double2 o = sacc[lane_row + (kRowsT / R) * r]; dsum[r] += o.x; dsq[r] += o.y; }
            }
        }
        if (part == 0) {
            double2* slot = static_cast<double2*>(p.part) +
                            (size_t)(2 * blockIdx.x + (c0 == 0 ? 1 : 0)) * kRowsT + lane_row;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = row0 + lane_row + (kRowsT / R) * r;
                if (n != p.col_tiles) slot[(kRowsT / R) * r] = make_double2(dsum[r], dsq[r]);
                else if (i < p.Nrow) {
                    p.Y[i] = (float)(dsum[r] * (p.left ? (double)p.left[i] : 1.0));
                    if (p.rowsq) p.rowsq[i] = dsq[r];
                }
            }
        }
    }
    grid_go();
}

// Finishes the row tiles that a cut falls into.  Block = (32 rows of a row tile, 8 columns), 8 groups of shares read in parallel (a row
// tile of a small problem has up to a hundred).  Every block waits for the product, also one that has nothing to add: what follows
// this kernel in the stream waits for this kernel only.
constexpr int kFixCols = 8;
__global__ void __launch_bounds__(256)
k_direct_fix(const DirectParams p, int BT, int ctas) {
    __shared__ float sm[kFixCols][8][32];
    const int rt = blockIdx.x / (kRowsT / 32);
    const long long total = (long long)p.row_tiles * p.col_tiles;
    const long long g0 = (long long)rt * p.col_tiles;
    const long long g1 = g0 + p.col_tiles;
    // the last CTA whose range begins at or before step g0, and the last one whose range begins before g1
    const int first = (int)(((g0 + 1) * ctas - 1) / total), last = (int)((g1 * ctas - 1) / total);
    grid_wait();
    grid_go();
    if (first == last) return;                                         // not cut: its CTA stored it
    const int r = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int row = (blockIdx.x % (kRowsT / 32)) * 32 + r, col0 = (int)blockIdx.y * kFixCols;
    const int per = (last - first + 8) / 8, s0 = first + grp * per, s1 = min(last + 1, s0 + per);
    const float* slots = static_cast<const float*>(p.part) + (size_t)col0 * kRowsT + row;
    float v[kFixCols];
#pragma unroll
    for (int c = 0; c < kFixCols; ++c) v[c] = 0.f;
#pragma unroll 4
    for (int s = s0; s < s1; ++s) {
        const float* o = slots + (size_t)(2 * s + (s == first ? 1 : 0)) * BT * kRowsT;
#pragma unroll
        for (int c = 0; c < kFixCols; ++c)
            if (col0 + c < p.b) v[c] += o[c * kRowsT];
    }
#pragma unroll
    for (int c = 0; c < kFixCols; ++c) sm[c][grp][r] = v[c];
    __syncthreads();
    // group g finishes column col0 + g
    const int64_t i = (int64_t)rt * kRowsT + row;
    if (i >= p.Nrow || col0 + grp >= p.b) return;
    float x = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) x += sm[grp][q][r];
    p.Y[i + (int64_t)(col0 + grp) * p.ldy] = x * (p.left ? p.left[i] : 1.0f);
}

// The same for row sums: block = 32 rows.
__global__ void __launch_bounds__(256)
k_direct_rowsum_fix(const DirectParams p, int ctas) {
    __shared__ double2 sm[8][32];
    const int rt = blockIdx.x / (kRowsT / 32);
    const long long total = (long long)p.row_tiles * p.col_tiles;
    const long long g0 = (long long)rt * p.col_tiles;
    const long long g1 = g0 + p.col_tiles;
    const int first = (int)(((g0 + 1) * ctas - 1) / total), last = (int)((g1 * ctas - 1) / total);
    grid_wait();
    grid_go();
    if (first == last) return;
    const int r = threadIdx.x & 31, grp = threadIdx.x >> 5, row = (blockIdx.x % (kRowsT / 32)) * 32 + r;
    const int per = (last - first + 8) / 8, s0 = first + grp * per, s1 = min(last + 1, s0 + per);
    const double2* slots = static_cast<const double2*>(p.part) + row;
    double2 v = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int s = s0; s < s1; ++s) { const double2 o = slots[(size_t)(2 * s + (s == first ? 1 : 0)) * kRowsT]; v.x += o.x; v.y += o.y; }
    sm[grp][r] = v;
    __syncthreads();
    const int64_t i = (int64_t)rt * kRowsT + row;
    if (grp != 0 || i >= p.Nrow) return;
    v = make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < 8; ++q) { v.x += sm[q][r].x; v.y += sm[q][r].y; }
    if (p.rowsq) p.rowsq[i] = v.y;
    p.Y[i] = (float)(v.x * (p.left ? (double)p.left[i] : 1.0));
}

// Block mode of small problems: a cluster of eight CTAs per 64 rows, a CTA an eighth of the columns, a warp an eighth of those; the sums
// meet in shared memory, first the warps' of each CTA, then the CTAs' through the cluster.  One launch and no shares in memory: N = 2048 cut into
// 512 ranges of the kernel above writes 4 MB of them for a second kernel to add.
constexpr int kSmallRows = 64, kSmallThr = 256, kSmallCtas = 8;
template <int DP4, int BT>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThr)
k_direct_small(const DirectParams p) {
    grid_wait();
    grid_go();
    constexpr int BP = BT + 4, kWarps = kSmallThr / 32, R = kSmallRows / 32;
    constexpr int kStage = kSmallThr * (4 * DP4 + BP), kRed = kWarps * BT * kSmallRows;
    __shared__ __align__(16) float smem[kStage > kRed ? kStage : kRed];
    __shared__ float total[BT * kSmallRows];             // [column][row]
    float4* sx = reinterpret_cast<float4*>(smem);
    float* sw = smem + kSmallThr * 4 * DP4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = (int)blockIdx.x % kSmallCtas;
    const int64_t row0 = (int64_t)(blockIdx.x / kSmallCtas) * kSmallRows;
    const int64_t per = (p.N + kSmallCtas - 1) / kSmallCtas, j_end = per * (rank + 1) < p.N ? per * (rank + 1) : p.N;
    float4 xi[R][DP4];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = row0 + lane + 32 * r;
#pragma unroll
        for (int k = 0; k < DP4; ++k) xi[r][k] = i < p.Nrow ? p.xrow[i * DP4 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float sum[R][BT];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < BT; ++c) sum[r][c] = 0.f;
    for (int64_t j0 = per * rank; j0 < j_end; j0 += kSmallThr) {
        const int n = (int)(j_end - j0 < kSmallThr ? j_end - j0 : kSmallThr), t = threadIdx.x;
        __syncthreads();
        if (t < n) {
            float w[BT];
#pragma unroll
            for (int c = 0; c < BT; ++c) w[c] = c < p.b ? (c < p.vcols ? p.V[j0 + t + (int64_t)c * p.ldv] : 1.f) : 0.f;
            const float right = p.right ? p.right[j0 + t] : 1.f;
#pragma unroll
            for (int k = 0; k < DP4; ++k) sx[t * DP4 + k] = p.xcol[(j0 + t) * DP4 + k];
#pragma unroll
            for (int c = 0; c < BT; ++c) sw[t * BP + c] = w[c] * right;
        }
        __syncthreads();
        const int jj0 = n * warp / kWarps, jj1 = n * (warp + 1) / kWarps;
        // (sums of eight columns, then of those: neighbouring points' large values do not meet the far ones' small ones in one long sum)
        auto column = [&](Sums<R, BT>& acc, int jj) {
            float kij[R];
            kernel_values<DP4, R>(sx, jj, xi, p.nbeta2, kij);
            acc.add(kij, reinterpret_cast<const float4*>(&sw[jj * BP]));
        };
        int jj = jj0;
        while (jj < jj1) {
            Sums<R, BT> acc;
            acc.clear();
            if (jj + 8 <= jj1) {
#pragma unroll
                for (int u = 0; u < 8; ++u) column(acc, jj + u);
                jj += 8;
            } else {
#pragma unroll 1
                for (; jj < jj1; ++jj) column(acc, jj);
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < BT; ++c) sum[r][c] += acc.get(r, c);
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < BT; ++c) smem[(warp * BT + c) * kSmallRows + lane + 32 * r] = sum[r][c];
    __syncthreads();
    for (int e = threadIdx.x; e < BT * kSmallRows; e += kSmallThr) {
        float x = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) x += smem[w * BT * kSmallRows + e];
        total[e] = x;
    }
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    cluster.sync();
    // every CTA finishes an eighth of the 64 x BT sums
    for (int t = threadIdx.x; t < BT * kSmallRows / kSmallCtas; t += kSmallThr) {
        const int e = rank * (BT * kSmallRows / kSmallCtas) + t, c = e / kSmallRows;
        float v[kSmallCtas];
#pragma unroll
        for (int q = 0; q < kSmallCtas; ++q) v[q] = *cluster.map_shared_rank(&total[e], q);
        const int64_t i = row0 + e % kSmallRows;
        if (c < p.b && i < p.Nrow) {
            const float x = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
            p.Y[i + (int64_t)c * p.ldy] = x * (p.left ? p.left[i] : 1.0f);
        }
    }
    cluster.sync();                                      // (a CTA's sums stay until the others have read them)
}

// Launches one CTA per equal range of steps: as many as are resident at once (more would leave a last round partly filled), or as
// asked (option "splits": ranges per row tile), within the slots' capacity.
template <class Kernel>
fd_status launch(fd_ctx* c, Kernel kernel, int smem, int per_sm, int BT, DirectParams p) {
    // Column tiles of 16 where 64 would give fewer than four steps per CTA: with one or two, the ranges differ by a factor of two and
    // small problems leave SMs idle (N = 1000, b = 64: 29 -> 21 us); more steps make the two barriers per tile dearer.
    p.tj_log2 = ceil_div(p.N, kTJ) * p.row_tiles < 4ll * c->sm_count * per_sm ? 4 : 6;
    p.col_tiles = (int)ceil_div(p.N, (int64_t)1 << p.tj_log2);
    const long long total = (long long)p.row_tiles * p.col_tiles;
    const size_t slot_floats = (size_t)kRowsT * (BT > 0 ? BT : 4);
    long long ctas = c->opt_splits > 0 ? (long long)p.row_tiles * c->opt_splits : (long long)c->sm_count * per_sm;
    ctas = std::max<long long>(1, std::min<long long>(std::min(ctas, total), (long long)(c->L.part_floats / (2 * slot_floats))));
    if (c->opt_splits <= 0) ctas = ceil_div(total, ceil_div(total, ctas));      // same longest range, fewer shares
    if (smem > 48 * 1024) FD_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // (not behind the kernel before: CTAs placed while that one still holds some SMs are spread unevenly, and the ranges are equal; N = 10000, b = 4: 67 -> 78 us)
    kernel<<<(unsigned)ctas, kThr, smem, c->stream>>>(p);
    FD_LAUNCH_CHECK(c, "k_direct");
    bool cut = false;
    for (int i = 1; i < ctas && !cut; ++i) cut = range_begin(total, i, (int)ctas) % p.col_tiles != 0;
    if (cut) {
        // launched while the product's last CTAs run (it waits for their stores): the launch costs no gap
        const dim3 grid((unsigned)p.row_tiles * (kRowsT / 32), BT > 0 ? (unsigned)ceil_div(p.b, kFixCols) : 1u);
        if (BT > 0) FD_CUDA(c, launch_behind(c->stream, grid, dim3(256), 0, k_direct_fix, p, BT, (int)ctas));
        else FD_CUDA(c, launch_behind(c->stream, grid, dim3(256), 0, k_direct_rowsum_fix, p, (int)ctas));
        FD_LAUNCH_CHECK(c, "k_direct_fix");
    }
    return FD_OK;
}

// Largest set that goes to the cluster kernel.  Against the ranges above: N = 1000, b = 8: 18.0 -> 8.8 us; 2048: 15.5 -> 11.3; 4096: 25.5 -> 25.3; b = 16,
// N = 2048: 19.4 -> 11.7, 4096: 34.7 -> 36.5.
constexpr int64_t small_n(int BT) { return BT <= 8 ? 3072 : 2048; }

template <int DP4, int BT>
fd_status launch_block(fd_ctx* c, const DirectParams& p) {
    if constexpr (DP4 <= 2 && BT <= 16)
        if (p.N <= small_n(BT) && p.Nrow <= small_n(BT) && c->opt_splits <= 0) {
            FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)(kSmallCtas * ceil_div(p.Nrow, kSmallRows))), dim3(kSmallThr), 0, k_direct_small<DP4, BT>, p));
            FD_LAUNCH_CHECK(c, "k_direct_small");
            return FD_OK;
        }
    constexpr int R = 4 * DP4 + BT <= 32 ? 4 : 2, H = R * kThr / kRowsT;
    constexpr int smem = (kTJ * DP4 * 4 + kTJ * (BT + 4) + H * BT * kRowsT) * 4;
    static const int per_sm = resident(k_direct<DP4, BT, R>, smem, kMaxCtasPerSm);
    return launch(c, k_direct<DP4, BT, R>, smem, per_sm, BT, p);
}

template <int DP4>
fd_status launch_dp(fd_ctx* c, int BT, const DirectParams& p) {
    switch (BT) {
        case 0: {
            static const int per_sm = resident(k_direct_rowsum<DP4>, 0, kMaxCtasPerSm);
            return launch(c, k_direct_rowsum<DP4>, 0, per_sm, 0, p);
        }
        case 4: return launch_block<DP4, 4>(c, p);
        case 8: return launch_block<DP4, 8>(c, p);
        case 16: return launch_block<DP4, 16>(c, p);
        case 24: return launch_block<DP4, 24>(c, p);
        case 32: return launch_block<DP4, 32>(c, p);
        case 48: return launch_block<DP4, 48>(c, p);
        default: return launch_block<DP4, 64>(c, p);
    }
}

}  // namespace

fd_status apply_simt(fd_ctx* c, const ApplyArgs& a) {
    const Layout& L = c->L;
    const int DP4 = L.DP / 4;
    if (DP4 > 8) return fail(c, FD_ERR_UNSUPPORTED, "SIMT path covers D <= 32 (got %d)", L.D);
    DirectParams p{};
    p.xrow = reinterpret_cast<const float4*>(a.xrow); p.Nrow = a.Nrow;
    p.xcol = reinterpret_cast<const float4*>(c->xs()); p.N = L.N;
    p.nbeta2 = (float)(-a.beta * kLog2e);
    p.right = a.right; p.left = a.left; p.ldv = a.ldv; p.ldy = a.ldy;
    p.part = c->at<float>(L.part);
    p.row_tiles = (int)ceil_div(a.Nrow, kRowsT);
    const bool rowsum = a.V == nullptr;
    // passes over the context's whole point set may leave out tiles of pairs whose kernel value is exactly zero; the degree passes
    // decide (they wait for their sums anyway), products follow
    if (a.rows_are_ctx && a.xrow == c->xs() && a.Nrow == L.N && !c->sh.on && L.direct_lists) {
        const int kind = rowsum && a.rowsq ? 2 : 4;
        FD_TRY(note_capture(c));
        FD_TRY(tile_lists(c, a.beta, kind, a.decide));
        if (c->lists[2].on && c->lists[2].beta == a.beta) return apply_direct_listed(c, a, kind);
    }
    const int chunks = rowsum ? 1 : (int)ceil_div(a.b, 64), step = (int)ceil_div(a.b, chunks);
    for (int c0 = 0; c0 < a.b; c0 += step) {
        const int bc = std::min(step, a.b - c0), BT = rowsum ? 0 : pick_bt(bc);
        p.V = rowsum ? nullptr : a.V + (int64_t)c0 * a.ldv;
        p.vcols = (a.ones_last ? a.b - 1 : a.b) - c0;
        p.b = bc;
        p.Y = a.Y + (int64_t)c0 * a.ldy;
        p.rowsq = a.rowsq;
        switch (DP4) {
            case 1: FD_TRY(launch_dp<1>(c, BT, p)); break;
            case 2: FD_TRY(launch_dp<2>(c, BT, p)); break;
            case 3: FD_TRY(launch_dp<3>(c, BT, p)); break;
            case 4: FD_TRY(launch_dp<4>(c, BT, p)); break;
            case 5: FD_TRY(launch_dp<5>(c, BT, p)); break;
            case 6: FD_TRY(launch_dp<6>(c, BT, p)); break;
            case 7: FD_TRY(launch_dp<7>(c, BT, p)); break;
            default: FD_TRY(launch_dp<8>(c, BT, p)); break;
        }
    }
    return FD_OK;
}

}  // namespace fd
