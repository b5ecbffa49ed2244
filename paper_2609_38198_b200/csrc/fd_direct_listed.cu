// Direct-difference fp32 passes over tile lists: sum_j K_ij right_j V_jc (Eqs. 5-6) and the row sums of the degree passes, leaving out the
// 64 x 16 tiles of pairs whose kernel values are all exactly zero (fd_order.cu).  Up to 8 coordinates, from 16384 points on.
//
// Everything here is in the points' order: an ordered copy of the points (made with the order) and an ordered, scaled copy of the right
// block (made per product, two microseconds), so that the 16 points of a list entry and their right rows are one contiguous piece each.
// A WARP owns 64 rows, two a lane (up to 4 columns: four), and takes its entries through a ring of its own in shared memory (cp.async), without any
// barrier of the block: neighbouring warps need not agree on which tiles are near.  The flat sequence of (64 rows, entry) steps is cut
// into equal ranges, one per warp; shares of row groups that a cut falls into are added by k_near_fix in the order of the warps.
//
// What bounds it: instruction issue, 2 D + b + 2 FMA-pipe operations per pair (N = 16384, D = 4, b = 16: 76 % of the issue slots taken, FMA pipe 60 %).  Against
// steps of 256 rows x 64 points gathered through the order, by a whole block and from boxes alone: 2-torus, N = 16384, beta = 100, b = 16: 134 -> 69 us
// a product (0.34 -> 0.17 of the tiles), both degree passes 164 -> 125; beta = 30: 310 (all tiles; not worth lists then) -> 157; N = 65536,
// b = 32, beta = 100: 1805 -> 1046.  Error against float64: 1.75e-7 -> 1.32e-7, 1.43e-7 -> 1.48e-7 and 4.3e-7 -> 2.1e-7 (short first sums).
#include <algorithm>

#include "fd_direct.h"

namespace fd {

namespace {

using namespace direct;

constexpr int kWarps = kThr / 32;
constexpr int kRowsG = 64;       // rows of a group: two per lane, or four with the points of an entry shared by the two halves of the warp
constexpr int kEntry = 16;       // points of a list entry
constexpr int kRing = 3;         // entries in a warp's ring
constexpr int kMaxCtasPerSm = 8;     // (fewer where the room for the shares of cut row groups says so)

struct NearParams {
    const float4* x;             // ordered points, DP4 float4 each, padded to whole entries with points whose kernel values are 0
    const float* w;              // ordered right block, BT floats a point (row sums: one weight a point, or null)
    const float* left;           // may be null
    float* Y; int64_t ldy; int b;
    double* rowsq;               // row sums: sum_j K_ij^2 (may be null)
    void* part;                  // two slots per warp: shares of row groups that are cut
    const unsigned short* list; const unsigned int* offs;      // entries of group g at list[g * entries ..], steps before it offs[g]
    const int* perm;
    unsigned char* near;         // row sums: where to note the entries with a kernel value that is not zero (may be null)
    int64_t N;
    float nbeta2;
    int groups, entries;         // row groups, entries of a whole row of tiles
    // columns of the right block with an entry that is not finite (set by the packing): bad[c] = epoch
    unsigned int* bad; unsigned int epoch;
    // for those columns: the points and the right block as they are
    const float4* xs; const float* V; int64_t ldv; int vcols; const float* right; int dp4;
};

// (a range without steps would leave its slots as they were: no more ranges than steps)
__device__ __forceinline__ int ranges(const NearParams& p, int warps) { return (int)p.offs[p.groups] < warps ? (int)p.offs[p.groups] : warps; }
__device__ __forceinline__ long long range_begin(long long total, int warp, int warps) { return total * warp / warps; }

// Last row group that begins at or before step g (a group holds one step at least).
__device__ __forceinline__ int group_of(const NearParams& p, long long g, int lane) {
    int lo = 0, n = p.groups;
    while (n > 1) {
        const int step = (n + 31) / 32, at = lane * step;
        const int before = __popc(__ballot_sync(0xffffffffu, at < n && (long long)p.offs[lo + (at < n ? at : 0)] <= g));
        lo += (before - 1) * step;
        n = min(step, n - (before - 1) * step);
    }
    return lo;
}

// A warp's range, row group by row group.
struct Range {
    long long g, g_end;
    int grp = -1, c0 = 0, n = 0, full = 0;               // entries c0 .. c0 + n of the group's `full` ones
    __device__ __forceinline__ Range(const NearParams& p, int warp, int warps) {
        const long long total = (long long)p.offs[p.groups];
        warps = ranges(p, warps);
        g = warp < warps ? range_begin(total, warp, warps) : 0;
        g_end = warp < warps ? range_begin(total, warp + 1, warps) : 0;
    }
    __device__ __forceinline__ bool next(const NearParams& p, int lane) {
        if (g >= g_end) return false;
        if (grp < 0) grp = group_of(p, g, lane);
        else ++grp;
        c0 = (int)(g - (long long)p.offs[grp]);
        full = (int)(p.offs[grp + 1] - p.offs[grp]);
        n = (int)(full - c0 < g_end - g ? full - c0 : g_end - g);
        g += n;
        return true;
    }
};

// Copies entry `e` (its points, then WF4 float4 of right rows per point) into a ring slot.
template <int DP4, int WF4>
__device__ __forceinline__ void load_entry(const NearParams& p, int e, float4* slot, int lane) {
    const float4* x = p.x + (size_t)e * kEntry * DP4;
    const float4* w = reinterpret_cast<const float4*>(p.w) + (size_t)e * kEntry * WF4;
#pragma unroll
    for (int t0 = 0; t0 < kEntry * (DP4 + WF4); t0 += 32) {
        const int t = t0 + lane;
        if (t < kEntry * (DP4 + WF4)) copy16(slot + t, t < kEntry * DP4 ? x + t : w + (t - kEntry * DP4));
    }
}

// Row r of a lane: row + step r of the group.
template <int R> struct Rows {
    static constexpr int kHalves = R / 2, kStep = kRowsG / R, kPoints = kEntry / kHalves;
    int row, half;                                       // first row; which part of an entry's points
    __device__ __forceinline__ Rows(int lane) : row(lane % kStep), half(lane / kStep) {}
};
template <int DP4, int R>
__device__ __forceinline__ void load_rows(const NearParams& p, int grp, const Rows<R>& rows, float4 (&xi)[R][DP4]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < DP4; ++k) xi[r][k] = p.x[((size_t)grp * kRowsG + rows.row + rows.kStep * r) * DP4 + k];
}

// Runs body(entry, slot) over the entries of a range's part, with kRing - 1 of them in flight.
template <int DP4, int WF4, class Body>
__device__ __forceinline__ void for_entries(const NearParams& p, const Range& range, float4* ring, int lane, Body body) {
    constexpr int kSlot = kEntry * (DP4 + WF4);
    const unsigned short* list = p.list + (size_t)range.grp * p.entries + range.c0;
    int mine = lane < range.n ? (int)list[lane] : 0;           // entries of 32 consecutive steps, one per lane
    int ahead = 0;                                             // next step to load
    auto load = [&]() {
        if (ahead < range.n) {
            const int e = __shfl_sync(0xffffffffu, mine, ahead & 31);
            load_entry<DP4, WF4>(p, e, ring + (ahead % kRing) * kSlot, lane);
            ++ahead;
            if ((ahead & 31) == 0 && ahead < range.n) mine = ahead + lane < range.n ? (int)list[ahead + lane] : 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int s = 0; s < kRing - 1; ++s) load();
    for (int t = 0; t < range.n; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
        __syncwarp();                                          // the entry has landed; everybody is done with the slot that load() refills
        load();
        body(t, ring + (t % kRing) * kSlot);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
}

// Rows per lane: four up to 4 columns, where the reads of x_j and w_j from shared memory are a quarter of the instructions: sets on which boxes are as
// good as notes were slower than a step of 256 rows x 64 points by a whole block without it (N = 100000, b = 1: circle 1763 us there, 1900 with
// two rows, 1673 with four; a line in R^7 4339, 4657 and 4313).
constexpr int near_rows(int BT) { return BT <= 4 ? 4 : 2; }
// (resident CTAs asked for, by the registers that the rows and sums of a thread need; 4 columns: four CTAs with all eight points of a turn unrolled, six
// with four of them 1857 us)
constexpr int near_ctas(int BT) { return BT <= 4 ? 4 : BT <= 8 ? 6 : BT <= 24 ? 4 : BT <= 48 ? 3 : 2; }
// Points per turn of the inner loop: as many as leave the sums in registers.  48 columns: two, with three resident CTAs, instead of four with two (N = 100000,
// b = 40: line in R^7 17.4 -> 15.2 ms, circle 9.36 -> 8.79); 5 to 8 coordinates, 8 columns: 5.88 -> 5.55 ms.
constexpr int near_unroll(int DP4, int BT) { return BT <= 4 ? 8 : BT == 48 || (DP4 == 2 && (BT == 8 || BT == 16)) ? 2 : 4; }

// Y[i, c] = left_i sum_j K_ij w[j, c] for c < b <= BT.
template <int DP4, int BT>
__global__ void __launch_bounds__(kThr, near_ctas(BT))
k_near(const NearParams p) {
    grid_wait();
    grid_go();
    constexpr int R = near_rows(BT), WF4 = BT / 4, kSlot = kEntry * (DP4 + WF4);
    extern __shared__ __align__(16) float4 smem_near[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warp = (int)blockIdx.x * kWarps + wib, warps = (int)gridDim.x * kWarps;
    float4* ring = smem_near + wib * kRing * kSlot;
    const Rows<R> rows(lane);
    Range range(p, warp, warps);
    while (range.next(p, lane)) {
        float4 xi[R][DP4];
        load_rows<DP4, R>(p, range.grp, rows, xi);
        Sums<R, BT> acc;
        acc.clear();
        // Two-level sums: the points are in their order, so one long fp32 sum would add the far points' small values to the near ones' large sum and
        // drop them, always with the same sign.  Up to 16 columns the second level is in registers, for wider blocks in the warp's slot.
        constexpr bool kInRegs = BT <= 16;
        static_assert(kInRegs || R == 2, "four rows a lane: sums in registers only");
        constexpr int kFlush = kInRegs ? 2 * rows.kHalves : 8;     // entries between flushes: 32 points (64 to memory: 1046 -> 1127 us at N = 65536, b = 32)
        float sum[R][kInRegs ? BT : 1];
        if (kInRegs) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < (kInRegs ? BT : 1); ++c) sum[r][c] = 0.f;
        }
        // the warp's slot for a share of this kind; sums that restart on the way wait there too
        float* slot_out = static_cast<float*>(p.part) + (size_t)(2 * warp + (range.c0 == 0 ? 1 : 0)) * BT * kRowsG + rows.row;
        bool flushed = false;
        for_entries<DP4, WF4>(p, range, ring, lane, [&](int t, const float4* slot) {
            const float4* sx = slot + rows.half * rows.kPoints * DP4;
            const float4* sw = slot + kEntry * DP4 + rows.half * rows.kPoints * WF4;
#pragma unroll near_unroll(DP4, BT)
            for (int jj = 0; jj < rows.kPoints; ++jj) {
                float kij[R];
                kernel_values<DP4, R>(sx, jj, xi, p.nbeta2, kij);
                acc.add(kij, sw + jj * WF4);
            }
            if ((t + 1) % kFlush == 0 && t + 1 < range.n) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < BT; ++c) {
                        if constexpr (kInRegs) sum[r][c] += acc.get(r, c);
                        else {
                            float* s = slot_out + c * kRowsG + rows.kStep * r;
                            *s = flushed ? *s + acc.get(r, c) : acc.get(r, c);
                        }
                    }
                acc.clear();
                flushed = true;
            }
        });
        const bool whole = range.n == range.full;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            // (four rows a lane: each half of the warp finishes two of them, and gets its share of these from the other)
            const int r = R == 2 ? u : u + 2 * rows.half;
            const int64_t pos = (int64_t)range.grp * kRowsG + rows.row + rows.kStep * r;
            const bool valid = pos < p.N;
            const int64_t i = valid ? p.perm[pos] : 0;
            const float l = whole && p.left ? p.left[i] : 1.0f;
#pragma unroll
            for (int c = 0; c < BT; ++c)
                if (c < p.b) {
                    float a;
                    if constexpr (R == 4) {
                        const float lo = acc.get(u, c) + sum[u][c], hi = acc.get(u + 2, c) + sum[u + 2][c];
                        a = (rows.half ? hi : lo) + __shfl_xor_sync(0xffffffffu, rows.half ? lo : hi, 16);
                    } else {
                        a = acc.get(u, c);
                        if constexpr (kInRegs) a += sum[u][c];
                        else if (flushed) a += slot_out[c * kRowsG + rows.kStep * r];
                    }
                    if (!whole) slot_out[c * kRowsG + rows.kStep * r] = a;
                    else if (valid) p.Y[i + (int64_t)c * p.ldy] = a * l;
                }
        }
    }
}

// sum_j K_ij w_j and sum_j K_ij^2; an entry (16 terms) in fp32, across entries in fp64.
template <int DP4, bool WEIGHTED>
__global__ void __launch_bounds__(kThr, 8)
k_near_rowsum(const NearParams p) {
    grid_wait();
    grid_go();
    constexpr int kSlot = kEntry * DP4;
    __shared__ float4 ring_store[kWarps * kRing * kSlot];
    constexpr int kRows = 2;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warp = (int)blockIdx.x * kWarps + wib, warps = (int)gridDim.x * kWarps;
    float4* ring = ring_store + wib * kRing * kSlot;
    Range range(p, warp, warps);
    while (range.next(p, lane)) {
        float4 xi[kRows][DP4];
        load_rows<DP4, kRows>(p, range.grp, Rows<kRows>(lane), xi);
        double dsum[kRows], dsq[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) { dsum[r] = 0.0; dsq[r] = 0.0; }
        const unsigned short* list = p.list + (size_t)range.grp * p.entries + range.c0;
        for_entries<DP4, 0>(p, range, ring, lane, [&](int t, const float4* slot) {
            const int e = (WEIGHTED || p.near) ? (int)__ldg(list + t) : 0;
            const float4* w4 = reinterpret_cast<const float4*>(p.w + (size_t)e * kEntry);
            float a[kRows], q[kRows];
#pragma unroll
            for (int r = 0; r < kRows; ++r) { a[r] = 0.f; q[r] = 0.f; }
#pragma unroll
            for (int j4 = 0; j4 < kEntry / 4; ++j4) {
                float4 w = make_float4(1.f, 1.f, 1.f, 1.f);
                if (WEIGHTED) w = __ldg(w4 + j4);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float kij[kRows];
                    kernel_values<DP4, kRows>(slot, 4 * j4 + u, xi, p.nbeta2, kij);
                    const float wj = u == 0 ? w.x : u == 1 ? w.y : u == 2 ? w.z : w.w;
#pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        a[r] = WEIGHTED ? fmaf(kij[r], wj, a[r]) : a[r] + kij[r];
                        q[r] = fmaf(kij[r], kij[r], q[r]);
                    }
                }
            }
            if (!WEIGHTED && p.near) {
                const bool any = __any_sync(0xffffffffu, a[0] + a[1] > 0.f);
                if (any && lane == 0) p.near[(size_t)range.grp * p.entries + e] = 1;
            }
#pragma unroll
            for (int r = 0; r < kRows; ++r) { dsum[r] += (double)a[r]; dsq[r] += (double)q[r]; }
        });
        const bool whole = range.n == range.full;
        double2* slot = static_cast<double2*>(p.part) + (size_t)(2 * warp + (range.c0 == 0 ? 1 : 0)) * kRowsG + lane;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const int64_t pos = (int64_t)range.grp * kRowsG + lane + 32 * r;
            if (!whole) slot[32 * r] = make_double2(dsum[r], dsq[r]);
            else if (pos < p.N) {
                const int64_t i = p.perm[pos];
                p.Y[i] = (float)(dsum[r] * (p.left ? (double)p.left[i] : 1.0));
                if (p.rowsq) p.rowsq[i] = dsq[r];
            }
        }
    }
}

// Row i's sum over every point for column c of the right block (row sums, V null: for the weights).  For columns that `bad` names: the product
// of an entry that is not finite with a kernel value of zero is NaN, so tiles of zeros count as well and the lists do not hold.
__device__ __forceinline__ float sum_over_all_points(const NearParams& p, int64_t i, int c) {
    float acc = 0.f;
#pragma unroll 1
    for (int64_t j = 0; j < p.N; ++j) {
        float h = 0.f;
#pragma unroll 1
        for (int k = 0; k < p.dp4; ++k) {
            const float4 a = p.xs[i * p.dp4 + k], b = p.xs[j * p.dp4 + k];
            const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
            h = fmaf(d0, d0, h); h = fmaf(d1, d1, h); h = fmaf(d2, d2, h); h = fmaf(d3, d3, h);
        }
        float w = p.V && c < p.vcols ? p.V[j + (int64_t)c * p.ldv] : 1.f;
        if (p.right) w *= p.right[j];
        acc = fmaf(ex2_approx(h * p.nbeta2), w, acc);
    }
    return acc;
}

// Finishes the row groups that a cut falls into, and the columns that `bad` names.  Block = (32 rows of a group, 8 columns), 8 groups of
// shares read in parallel.  Every block waits for the product, also one that has nothing to add: what follows this kernel in the
// stream waits for this kernel only.  ROWSUM: one column of (sum, sum of squares) in fp64.
constexpr int kFixCols = 8;
template <bool ROWSUM>
__global__ void __launch_bounds__(256)
k_near_fix(const NearParams p, int BT, int warps) {
    grid_wait();
    grid_go();
    __shared__ float sm[kFixCols][8][32];
    __shared__ double2 sd[8][32];
    const int grp = blockIdx.x / (kRowsG / 32);
    const long long total = (long long)p.offs[p.groups], g0 = (long long)p.offs[grp], g1 = (long long)p.offs[grp + 1];
    warps = ranges(p, warps);
    // the last warp whose range begins at or before step g0, and the last one whose range begins before g1
    const int first = (int)(((g0 + 1) * warps - 1) / total), last = (int)((g1 * warps - 1) / total);
    const bool cut = first != last;                                    // else its warp stored it
    const int r = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const int row = (blockIdx.x % (kRowsG / 32)) * 32 + r, col0 = (int)blockIdx.y * kFixCols;
    // (read beside the shares, looked at after them: one latency)
    const int col = ROWSUM ? 0 : col0 + sub;
    const unsigned int note = p.bad && col < p.b ? p.bad[col] : p.epoch + 1;
    if (cut) {
        const int per = (last - first + 8) / 8, s0 = first + sub * per, s1 = min(last + 1, s0 + per);
        if (ROWSUM) {
            const double2* slots = static_cast<const double2*>(p.part) + row;
            double2 v = make_double2(0.0, 0.0);
#pragma unroll 4
            for (int s = s0; s < s1; ++s) { const double2 o = slots[(size_t)(2 * s + (s == first ? 1 : 0)) * kRowsG]; v.x += o.x; v.y += o.y; }
            sd[sub][r] = v;
        } else {
            const float* slots = static_cast<const float*>(p.part) + (size_t)col0 * kRowsG + row;
            float v[kFixCols];
#pragma unroll
            for (int c = 0; c < kFixCols; ++c) v[c] = 0.f;
#pragma unroll 4
            for (int s = s0; s < s1; ++s) {
                const float* o = slots + (size_t)(2 * s + (s == first ? 1 : 0)) * BT * kRowsG;
#pragma unroll
                for (int c = 0; c < kFixCols; ++c)
                    if (col0 + c < p.b) v[c] += o[c * kRowsG];
            }
#pragma unroll
            for (int c = 0; c < kFixCols; ++c) sm[c][sub][r] = v[c];
        }
        __syncthreads();
    }
    const int64_t pos = (int64_t)grp * kRowsG + row;
    if (pos >= p.N || (ROWSUM ? sub != 0 : col >= p.b)) return;
    const bool bad = note == p.epoch;
    if (!cut && !bad) return;
    const int64_t i = p.perm[pos];
    if (ROWSUM) {
        double2 v = make_double2(0.0, 0.0);
        if (cut) {
#pragma unroll
            for (int q = 0; q < 8; ++q) { v.x += sd[q][r].x; v.y += sd[q][r].y; }
            if (p.rowsq) p.rowsq[i] = v.y;
        }
        if (bad) v.x = (double)sum_over_all_points(p, i, 0);
        p.Y[i] = (float)(v.x * (p.left ? (double)p.left[i] : 1.0));
    } else {
        float x = 0.f;
        if (bad) x = sum_over_all_points(p, i, col);
        else {
#pragma unroll
            for (int q = 0; q < 8; ++q) x += sm[sub][q][r];
        }
        p.Y[i + (int64_t)col * p.ldy] = x * (p.left ? p.left[i] : 1.0f);
    }
}

// w[pos * BT + c] = right_i V[i, c] for the point i at position pos, 0 beyond the points and the columns; a thread per four columns
// (row sums: BT = 1, a thread per four positions).  Notes the columns with an entry that is not finite.
__global__ void __launch_bounds__(256)
k_near_pack(const float* __restrict__ V, int64_t ldv, int vcols, const float* __restrict__ right, const int* __restrict__ perm, int64_t N, int64_t NP, int b, int BT,
            float4* __restrict__ w, unsigned int* __restrict__ bad, unsigned int epoch) {
    grid_wait();
    grid_go();
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const bool vec = BT == 1;
    const int per = vec ? 1 : BT / 4;
    const int64_t first = vec ? 4 * t : t / per;
    if (first >= NP) return;
    const int c0 = vec ? 0 : 4 * (int)(t % per);
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t pos = vec ? first + u : first;
        const int c = vec ? 0 : c0 + u;
        v[u] = 0.f;
        if (pos < N && c < b) {
            const int64_t i = perm[pos];
            float x = V && c < vcols ? V[i + (int64_t)c * ldv] : 1.f;
            if (right) x *= right[i];
            if (!isfinite(x)) bad[c] = epoch;
            v[u] = x;
        }
    }
    w[t] = make_float4(v[0], v[1], v[2], v[3]);
}

template <class Kernel>
fd_status launch(fd_ctx* c, Kernel kernel, int smem, int per_sm, int BT, NearParams p) {
    const size_t slot_floats = (size_t)kRowsG * (BT > 0 ? BT : 4);
    long long ctas = c->opt_splits > 0 ? ceil_div(p.N, 256) * c->opt_splits : (long long)c->sm_count * per_sm;
    ctas = std::max<long long>(1, std::min<long long>(ctas, (long long)(c->L.part_floats / (2 * kWarps * slot_floats))));
    const int warps = (int)ctas * kWarps;
    if (smem > 48 * 1024) FD_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // (behind the packing: N = 16384, D = 4, b = 16: 69.8 -> 68.0 us a product, launched after it and behind it)
    FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)ctas), dim3(kThr), smem, kernel, p));
    FD_LAUNCH_CHECK(c, "k_near");
    FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)p.groups * (kRowsG / 32), BT > 0 ? (unsigned)ceil_div(p.b, kFixCols) : 1u), dim3(256), 0,
                             BT > 0 ? k_near_fix<false> : k_near_fix<true>, p, BT, warps));
    FD_LAUNCH_CHECK(c, "k_near_fix");
    return FD_OK;
}

template <int DP4, int BT>
fd_status launch_block(fd_ctx* c, const NearParams& p) {
    constexpr int smem = kWarps * kRing * kEntry * (DP4 + BT / 4) * 16;
    static const int per_sm = resident(k_near<DP4, BT>, smem, kMaxCtasPerSm);
    return launch(c, k_near<DP4, BT>, smem, per_sm, BT, p);
}
template <int DP4>
fd_status launch_dp(fd_ctx* c, int BT, const NearParams& p) {
    switch (BT) {
        case 0: {
            static const int plain = resident(k_near_rowsum<DP4, false>, 0, kMaxCtasPerSm), weighted = resident(k_near_rowsum<DP4, true>, 0, kMaxCtasPerSm);
            if (p.w) return launch(c, k_near_rowsum<DP4, true>, 0, weighted, 0, p);
            return launch(c, k_near_rowsum<DP4, false>, 0, plain, 0, p);
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

fd_status apply_direct_listed(fd_ctx* c, const ApplyArgs& a, int kind) {
    const Layout& L = c->L;
    const int DP4 = L.DP / 4, buf = kind == 4 ? 0 : 1;
    const bool rowsum = a.V == nullptr;
    NearParams p{};
    p.x = c->at<float4>(L.xord); p.N = L.N; p.nbeta2 = (float)(-a.beta * kLog2e);
    p.left = a.left; p.right = a.right; p.ldy = a.ldy; p.ldv = a.ldv;
    p.part = c->at<float>(L.part); p.xs = reinterpret_cast<const float4*>(c->xs()); p.dp4 = DP4;
    p.groups = (int)(L.NP / kRowsG); p.entries = (int)(L.NP / kEntry);
    p.list = c->at<unsigned short>(L.lists[buf]);
    p.offs = c->at<unsigned int>(L.list_counts[buf]) + 2 * p.groups;
    p.perm = c->at<int>(L.perm);
    unsigned int* bad = reinterpret_cast<unsigned int*>(c->at<char>(L.status) + 256);
    float* w = c->at<float>(L.wt_hi);                    // (the Gram-form kernels' block operands are packed for every product: BP x NP floats)
    // the first degree pass (squares, no weights) notes the entries that are not all zero
    if (rowsum && a.rowsq && !a.right && a.decide && !c->captured && (c->near_beta != a.beta || !c->near_direct)) {
        c->near_beta = -1.0;
        p.near = c->at<unsigned char>(L.near);
        FD_CUDA(c, cudaMemsetAsync(p.near, 0, (size_t)p.groups * p.entries, c->stream));
    }
    const int chunks = rowsum ? 1 : (int)ceil_div(a.b, 64), step = (int)ceil_div(a.b, chunks);
    for (int c0 = 0; c0 < a.b; c0 += step) {
        const int bc = std::min(step, a.b - c0), BT = rowsum ? 0 : pick_bt(bc);
        p.V = rowsum ? nullptr : a.V + (int64_t)c0 * a.ldv;
        p.vcols = (a.ones_last ? a.b - 1 : a.b) - c0;
        p.b = bc;
        p.Y = a.Y + (int64_t)c0 * a.ldy;
        p.rowsq = a.rowsq;
        if (!rowsum || a.right) {
            // (a replayed graph brings the same epoch again; what an earlier replay noted would cost time, not the result)
            p.epoch = ++c->direct_epoch;
            p.bad = bad;
            if (c->captured) FD_CUDA(c, cudaMemsetAsync(bad, 0, 64 * 4, c->stream));
            const int64_t threads = rowsum ? L.NP / 4 : L.NP * (BT / 4);
            FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)ceil_div(threads, 256)), dim3(256), 0, k_near_pack, p.V, p.ldv, p.vcols, p.right, p.perm,
                                     L.N, L.NP, bc, rowsum ? 1 : BT, reinterpret_cast<float4*>(w), bad, p.epoch));
            FD_LAUNCH_CHECK(c, "k_near_pack");
            p.w = w;
        }
        if (DP4 == 1) FD_TRY(launch_dp<1>(c, BT, p));
        else FD_TRY(launch_dp<2>(c, BT, p));
    }
    if (p.near) { c->near_beta = a.beta; c->near_direct = true; c->near_unproven = true; }
    return FD_OK;
}

}  // namespace fd
