// Symmetric half-work row sums on tcgen05 / TMEM: sums[i] = sum_j w_j K_ij (and sum_ij K_ij^2) for a whole data set from the tiles on or
// above the diagonal alone (K = K^T, Sec. 2.1).  The degree passes of an unsharded context.
//
// The S tile (fd_tc_block.cu: exponents from the Gram MMAs) is built with the points of the STREAMED tile J on the TMEM lanes
// and the points of a CTA's resident tile It on the columns, so a thread owns one streamed point:
//   * its sum over the columns is that point's share of tile (J, It);
//   * acc[c] += w_J P[., c] collects, over the whole sweep, the resident point c's sum over the streamed points that fall on this
//     lane; the lanes are reduced (butterfly of shuffles) only every kSymFlush tiles, which also bounds the fp32 accumulation length.
// J < It is the mirror of a tile another resident tile evaluates (skipped: only the first streamed tile of the second resident tile);
// J == It counts once (resident side only); J > It counts for both sides.  The left weight is applied to the finished
// sums.  (Weights in the exponent would move it away from zero, where the tensor core's rounding of it differs from
// the one the block product sees, and the two would no longer cancel in diag(s) K diag(s).)  Sums go to one 64-bit
// fixed-point integer per point: integer additions commute, so the result does not depend on the order in which CTAs arrive.
//
// One persistent CTA per SM, two resident tiles (256 points), 20 warps:
//   warps 0-15   four warpgroups: warpgroup k takes columns [64 (k & 1), + 64) of resident tile k >> 1 (64 accumulators per thread);
//   warp 16      TMA producer (4-stage ring); warp 17 Gram-MMA issuer (four S buffers);
//   warps 18, 19 collectors: add the four partial sums of a streamed point (two resident tiles x two column halves) from
//                shared memory, so that a pair of tiles costs one atomic per streamed point.
// Work is a flat sequence of (resident pair, streamed tile) steps, cut into equal ranges, one per CTA.
//
// What bounds it: the MUFU (1024 SM clocks per tile; 78 to 81 % busy at N = 65536) and the queue that feeds it, with the additions beside it (issue
// slots 53 to 55 %, 60 to 63 % with scalar additions).  The additions work on two columns an instruction (add / fma.rn.f32x2): half their issue slots, the same
// bits.  N = 65536: 1440 -> 1376 us both passes, N = 2^18: 21.55 -> 20.4 ms.  (Loads of 8 columns one step ahead: 1.5 % slower; a polynomial
// on the FMA pipe for two of sixteen columns: 4 % slower.)  Both degree passes at N = 2^18 (one with squares, one
// with weights), scalar: 26.2 -> 21.6 ms against two warpgroups with 128 accumulators a thread, whole row pairs per CTA and an atomic per
// point and tile.
#include <algorithm>
#include <cmath>

#include "fd_tc_common.h"

namespace fd {

namespace {

using namespace tc;

constexpr int kThreadsS = 640;
constexpr int kRegsLaunch = 96, kRegsExp = 104, kRegsUtil = 64;
static_assert(kThreadsS * kRegsLaunch == 512 * kRegsExp + 128 * kRegsUtil, "setmaxnreg must conserve the register total");
constexpr int kSymFlush = 64;          // tiles between reductions of the resident sums
constexpr int kXChunk = 128 * 64;      // one K slab (hi|lo) of 128 points: 8 KB
constexpr int kSlots = 4;              // ring of streamed partial sums
// 2^(bias - 40) and 2^(bias - 60), squared (a tenth below: the same value comes out of another kernel's accumulator as well)
constexpr float kNearProduct2 = 0.9f * 0x1p-50f, kNearSums2 = 0.9f * 0x1p-90f;

struct BarriersS {
    uint64_t full[kStages], empty[kStages];   // streamed tile: TMA -> Gram issuer -> TMA
    uint64_t xfull, xempty;                   // resident tiles
    uint64_t s_full[4], s_done[4];            // [S buffer]: exponent tile ready / in registers (8 warps)
    uint64_t r_ready[kSlots], r_free[kSlots]; // partial sums of a streamed tile written (16 warps) / collected (2 warps)
    double sq[16];
    uint32_t tmem_base;
    int abort_flag;
};

struct SymParams {
    int64_t N, np;
    unsigned long long* sums;    // N fixed-point sums, units of 2^-shift (of the 2^bias-scaled kernel values)
    double* sq;                  // per CTA: its share of sum_ij K_ij^2 (null: not wanted)
    const float* weights;        // padded right weights (weighted instantiation)
    unsigned int* status;
    int pairs, num_jt, K16, shift;
    // tile lists (null: every tile): the streamed tiles of resident pair r are the last uoffs[r + 1] - uoffs[r] entries of its list
    const unsigned short* list; const unsigned int* counts; const unsigned int* uoffs;
    // notes of the tiles that hold a value of the product's / the row sums' range, num_jt x num_jt bytes each (null: not wanted)
    unsigned char* near_product; unsigned char* near_sums;
};

constexpr int smem_total(int K16) { return 1024 + kStages * K16 * kXChunk + 2 * K16 * kXChunk + kSlots * 4 * 128 * 4 + 1024; }

// Steps before resident pair r: pair r has the streamed tiles 2 r .. num_jt - 1.
__host__ __device__ __forceinline__ long long steps_before(long long r, long long num_jt) { return r * num_jt - r * (r - 1); }
// A CTA's range, item by item.  One type without lists and one with them: the exponential warps of the weighted instantiation
// have no register to spare (scalar sums: one type with a run-time choice spilled 176 B a thread instead of 28: N = 2^18, both passes 21.7 ->
// 23.0 ms; with packed sums the weighted instantiations spill 36 and, with lists, 44 B, those with squares 12).
template <bool LISTED> struct Item;
template <> struct Item<false> {
    int pair, j0, n;             // streamed tiles j0 ..
    __device__ __forceinline__ int tile(const SymParams&, int j) const { return j0 + j; }
};
template <> struct Item<true> {
    int pair, first, n;          // entries first .. of the lists
    __device__ __forceinline__ int tile(const SymParams& p, int j) const { return (int)__ldg(p.list + (first + j)); }
};
template <bool LISTED> struct Steps;
template <> struct Steps<false> {
    int pair, j, left, num_jt;
    __device__ __forceinline__ Steps(const SymParams& p) {
        const long long total = steps_before(p.pairs, p.num_jt);
        const long long g0 = total * blockIdx.x / gridDim.x, g1 = total * (blockIdx.x + 1) / gridDim.x;
        num_jt = p.num_jt;
        // largest r with steps_before(r) <= g0
        const double h = 0.5 * (num_jt + 1.0);
        long long r = (long long)(h - sqrt(fmax(0.0, h * h - (double)g0)));
        r = r < 0 ? 0 : r >= p.pairs ? p.pairs - 1 : r;
        while (r > 0 && steps_before(r, num_jt) > g0) --r;
        while (r + 1 < p.pairs && steps_before(r + 1, num_jt) <= g0) ++r;
        pair = (int)r;
        j = 2 * pair + (int)(g0 - steps_before(r, num_jt));
        left = (int)(g1 - g0);
    }
    __device__ __forceinline__ bool next(const SymParams&, Item<false>& it) {
        if (left <= 0) return false;
        it.pair = pair; it.j0 = j;
        it.n = num_jt - j < left ? num_jt - j : left;
        left -= it.n; ++pair; j = 2 * pair;
        return true;
    }
};
template <> struct Steps<true> {
    int pair, done, left;        // `done` steps of the pair lie before the range
    __device__ __forceinline__ Steps(const SymParams& p) {
        const long long total = (long long)p.uoffs[p.pairs];
        const long long g0 = total * blockIdx.x / gridDim.x, g1 = total * (blockIdx.x + 1) / gridDim.x;
        int lo = 0, hi = p.pairs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((long long)p.uoffs[mid] <= g0) lo = mid;
            else hi = mid - 1;
        }
        pair = lo;
        done = (int)(g0 - (long long)p.uoffs[pair]);
        left = (int)(g1 - g0);
    }
    __device__ __forceinline__ bool next(const SymParams& p, Item<true>& it) {
        if (left <= 0) return false;
        const int full = (int)(p.uoffs[pair + 1] - p.uoffs[pair]);
        it.pair = pair;
        it.first = pair * p.num_jt + (int)p.counts[pair] - full + done;
        it.n = full - done < left ? full - done : left;
        left -= it.n; ++pair; done = 0;
        return true;
    }
};

template <bool SQ, bool WEIGHTED, bool LISTED, bool NOTED>
__global__ void __launch_bounds__(kThreadsS, 1)
k_sym(const __grid_constant__ CUtensorMap map_res, const __grid_constant__ CUtensorMap map_str, const SymParams p) {
    extern __shared__ uint8_t smem_raw[];
    const int K16 = p.K16;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_base = base;
    uint8_t* xi_base = base + kStages * K16 * kXChunk;                        // 2 resident tiles x K16 slabs
    float* rbuf = reinterpret_cast<float*>(xi_base + 2 * K16 * kXChunk);      // [slot][resident tile, column half][128 streamed points]
    BarriersS* bars = reinterpret_cast<BarriersS*>(rbuf + kSlots * 4 * 128);
    volatile int* abort_flag = &bars->abort_flag;
    const int warp = warp_index(), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
        mbar_init(&bars->xfull, 1); mbar_init(&bars->xempty, 1);
        for (int u = 0; u < 4; ++u) { mbar_init(&bars->s_full[u], 1); mbar_init(&bars->s_done[u], 8); }
        for (int u = 0; u < kSlots; ++u) { mbar_init(&bars->r_ready[u], 16); mbar_init(&bars->r_free[u], 2); }
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    const long long t_begin = clock64();

    if (warp >= 16) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsUtil));
      if (warp == 16) {
        // =============================================================== TMA producer (one thread)
        if (elect_one()) {
            prefetch_tmap(&map_res); prefetch_tmap(&map_str);
            uint32_t k = 0, xph = 1;                               // step counter; parity of the resident tiles' "empty" phase
            bool ok = true;
            Steps<LISTED> steps(p);
            for (Item<LISTED> it; ok && steps.next(p, it);) {
                ok = mbar_wait(&bars->xempty, xph, abort_flag, p.status, 1);
                if (!ok) break;
                xph ^= 1u;
                mbar_expect_tx(&bars->xfull, 2 * K16 * kXChunk);
                for (int t = 0; t < 2; ++t)
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(xi_base + (t * K16 + c) * kXChunk, &map_res, 0, (int)(c * p.np + (int64_t)it.pair * 256 + t * 128), &bars->xfull);
                for (int j = 0; j < it.n; ++j, ++k) {
                    const uint32_t s = k % kStages;
                    ok = mbar_wait(&bars->empty[s], ((k / kStages) & 1) ^ 1, abort_flag, p.status, 2);
                    if (!ok) break;
                    mbar_expect_tx(&bars->full[s], K16 * kXChunk);
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(stage_base + (s * K16 + c) * kXChunk, &map_str, 0, (int)(c * p.np + (int64_t)it.tile(p, j) * 128), &bars->full[s]);
                }
            }
            if (!ok) {
                // aborted: let the copies already in flight land before the CTA exits (bounded)
                for (uint32_t i = (k > (uint32_t)kStages ? k - kStages : 0); i < k; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(&bars->full[i % kStages], (i / kStages) & 1) && clock64() - t0 < 20000000ll) {}
                }
            }
        }
      } else if (warp == 17) {
        // =============================================================== Gram MMA issuer (one thread)
        if (elect_one()) {
            constexpr uint32_t idesc_g = idesc_f16(128);
            const uint64_t xd = smem_desc(smem_u32(xi_base), 512, 4);      // 64 B rows (SWIZZLE_64B), 512 B between 8-row groups
            const uint32_t xi_lo = (uint32_t)xd, xdesc_hi = (uint32_t)(xd >> 32);
            const uint32_t stage_lo = (uint32_t)smem_desc(smem_u32(stage_base), 512, 4);
            constexpr uint32_t kSlab = kXChunk >> 4;
            uint32_t k = 0, xph = 0;
            bool ok = true;
            Steps<LISTED> steps(p);
            for (Item<LISTED> it; ok && steps.next(p, it);) {
                ok = mbar_wait(&bars->xfull, xph, abort_flag, p.status, 3);
                if (!ok) break;
                xph ^= 1u;
                for (int j = 0; j < it.n && ok; ++j, ++k) {
                    const uint32_t s = k % kStages;
                    ok = mbar_wait(&bars->full[s], (k / kStages) & 1, abort_flag, p.status, 4);
                    if (!ok) break;
                    for (uint32_t t = 0; t < 2; ++t) {
                        const uint32_t buf = (2 * k + t) & 3;
                        ok = mbar_wait(&bars->s_done[buf], ((k >> 1) & 1) ^ 1, abort_flag, p.status, 5);
                        if (!ok) break;
                        tc_fence_after();
                        // The streamed tile is the M operand.  The two small cross terms (hi x lo) go first and the large hi x hi
                        // term last: each MMA rounds its result at the magnitude of its largest addend.
                        const uint32_t s_addr = tmem + 128u * buf;
                        const uint32_t a0 = stage_lo + s * (uint32_t)K16 * kSlab, b0 = xi_lo + t * (uint32_t)K16 * kSlab;
                        for (int c = 0; c < K16; ++c) {
                            const uint32_t a = a0 + (uint32_t)c * kSlab, b = b0 + (uint32_t)c * kSlab;
                            if (c == 0) mma_ss2<0>(s_addr, a, xdesc_hi, b + 2, xdesc_hi, idesc_g);      // + 2: the lo half starts 32 B into the row
                            else mma_ss2<1>(s_addr, a, xdesc_hi, b + 2, xdesc_hi, idesc_g);
                            mma_ss2<1>(s_addr, a + 2, xdesc_hi, b, xdesc_hi, idesc_g);
                        }
                        for (int c = 0; c < K16; ++c)
                            mma_ss2<1>(s_addr, a0 + (uint32_t)c * kSlab, xdesc_hi, b0 + (uint32_t)c * kSlab, xdesc_hi, idesc_g);
                        tc_commit(&bars->s_full[buf]);
                    }
                    if (!ok) break;
                    tc_commit(&bars->empty[s]);
                }
                if (ok) tc_commit(&bars->xempty);                  // the resident tiles may be replaced
            }
        }
      } else {
        // =============================================================== collectors: 64 streamed points each, two per lane
        const double fix = (double)(1ull << p.shift);
        const int pt0 = (warp - 18) * 64 + lane * 2;
        uint32_t k = 0;
        bool ok = true;
        Steps<LISTED> steps(p);
        for (Item<LISTED> it; ok && steps.next(p, it);) {
            for (int j = 0; j < it.n; ++j, ++k) {
                const uint32_t slot = k % kSlots;
                ok = mbar_wait(&bars->r_ready[slot], (k / kSlots) & 1, abort_flag, p.status, 12);
                if (!ok) break;
                const float2* r = reinterpret_cast<const float2*>(rbuf + slot * 512 + pt0);
                const float2 a = r[0], b = r[64], c = r[128], d = r[192];
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->r_free[slot]);
                const float x = (a.x + b.x) + (c.x + d.x), y = (a.y + b.y) + (c.y + d.y);
                const int64_t pt = (int64_t)it.tile(p, j) * 128 + pt0;
                if (pt < p.N && x != 0.f) atomicAdd(p.sums + pt, (unsigned long long)__double2ll_rn((double)x * fix));
                if (pt + 1 < p.N && y != 0.f) atomicAdd(p.sums + pt + 1, (unsigned long long)__double2ll_rn((double)y * fix));
            }
        }
      }
    } else {
        // =============================================================== exponential warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsExp));
        const int wg = warp >> 2, t = wg >> 1, h = wg & 1, wq = warp & 3;
        const uint32_t addr0 = tmem + ((uint32_t)(wq * 32) << 16) + 64u * h;
        const int pt_in_tile = wq * 32 + lane;
        uint32_t k = 0;
        double dsq = 0.0;
        bool ok = true;
        uint64_t acc2[32];                                         // two columns each
        Steps<LISTED> steps(p);
        for (Item<LISTED> it; ok && steps.next(p, it);) {
            const int It = 2 * it.pair + t;
            const ulonglong2* wres = WEIGHTED ? reinterpret_cast<const ulonglong2*>(p.weights + (int64_t)It * 128 + 64 * h) : nullptr;
#pragma unroll
            for (int c = 0; c < 32; ++c) acc2[c] = 0;
            int pending = 0;                                       // tiles accumulated in acc since the last reduction
            for (int j = 0; j < it.n; ++j, ++k) {
                const int J = it.tile(p, j);
                const float wj = WEIGHTED ? __ldg(p.weights + (int64_t)J * 128 + pt_in_tile) : 1.f;
                const uint64_t wj2 = pair2(wj, wj);
                const uint32_t buf = (2 * k + (uint32_t)t) & 3;
                ok = mbar_wait(&bars->s_full[buf], (k >> 1) & 1, abort_flag, p.status, 8);
                if (!ok) break;
                tc_fence_after();
                const bool use = J >= It;
                uint64_t r2 = 0, q2 = 0;
                if (use) {
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        uint32_t sv[16];
                        tmem_ld16(addr0 + 128u * buf + 16 * ch, sv);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; i += 4) {
                            ulonglong2 w4;
                            if (WEIGHTED) w4 = __ldg(wres + 4 * ch + i / 4);
#pragma unroll
                            for (int u = 0; u < 4; u += 2) {
                                uint64_t& a = acc2[(16 * ch + i + u) / 2];
                                const uint64_t p2 = pair2(ex2f(__uint_as_float(sv[i + u])), ex2f(__uint_as_float(sv[i + u + 1])));
                                if (WEIGHTED) { a = fma2(p2, wj2, a); r2 = fma2(p2, u ? w4.y : w4.x, r2); }
                                else { a = add2(a, p2); r2 = add2(r2, p2); }
                                if (SQ) q2 = fma2(p2, p2, q2);
                            }
                        }
                    }
                }
                // the buffer can be refilled: its values are in registers or consumed
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->s_done[buf]);
                const bool both = J > It;                          // off the diagonal: counts for the streamed side too
                const uint32_t slot = k % kSlots;
                ok = mbar_wait(&bars->r_free[slot], ((k / kSlots) & 1) ^ 1, abort_flag, p.status, 13);
                if (!ok) break;
                const float2 rp = split2(r2);
                const float r = rp.x + rp.y;
                rbuf[slot * 512 + wg * 128 + pt_in_tile] = both ? r : 0.f;
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->r_ready[slot]);
                if (SQ && use) {
                    const float2 qp = split2(q2);
                    const float q = qp.x + qp.y;
                    dsq += (double)q * (both ? 2.0 : 1.0);
                    if (NOTED) {
                        // a value at or above a limit shows in its thread's sum of squares
                        const bool sums = __any_sync(0xffffffffu, q >= kNearSums2), product = __any_sync(0xffffffffu, q >= kNearProduct2);
                        if (lane == 0 && sums) {
                            const size_t a = (size_t)It * p.num_jt + J, b = (size_t)J * p.num_jt + It;
                            p.near_sums[a] = 1; p.near_sums[b] = 1;
                            if (product) { p.near_product[a] = 1; p.near_product[b] = 1; }
                        }
                    }
                }
                if (use) ++pending;
                if (pending == kSymFlush || (j + 1 == it.n && pending > 0)) {
                    // sums of acc over the 32 lanes: lane l ends up with columns l and 32 + l
                    const double fix = (double)(1ull << p.shift);
                    float acc[64];
#pragma unroll
                    for (int c = 0; c < 32; ++c) { const float2 a = split2(acc2[c]); acc[2 * c] = a.x; acc[2 * c + 1] = a.y; }
#pragma unroll
                    for (int ch = 0; ch < 2; ++ch) {
#pragma unroll
                        for (int m = 16; m >= 1; m >>= 1) {
                            const bool up = (lane & m) != 0;
#pragma unroll
                            for (int q = 0; q < m; ++q) {
                                const float send = up ? acc[32 * ch + q] : acc[32 * ch + q + m];
                                const float keep = up ? acc[32 * ch + q + m] : acc[32 * ch + q];
                                acc[32 * ch + q] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                            }
                        }
                        const int64_t pt = (int64_t)It * 128 + 64 * h + 32 * ch + lane;
                        if (pt < p.N) atomicAdd(p.sums + pt, (unsigned long long)__double2ll_rn((double)acc[32 * ch] * fix));
                    }
#pragma unroll
                    for (int c = 0; c < 32; ++c) acc2[c] = 0;
                    pending = 0;
                }
            }
        }
        if (SQ) {
#pragma unroll
            for (int m = 16; m >= 1; m >>= 1) dsq += __shfl_xor_sync(0xffffffffu, dsq, m);
            if (lane == 0) bars->sq[warp] = dsq;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (SQ && threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < 16; ++w) a += bars->sq[w];
        p.sq[blockIdx.x] = a * (1.0 / ((double)(1 << kBias) * (double)(1 << kBias)));
    }
    // SM cycles CTA 0 spent on its work items (status words 2-3): lets the host relate the kernel time to the SM clock
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<long long*>(p.status + 2) = clock64() - t_begin;
    if (warp == 16) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Fixed-point sums -> q (times the left weight); clears the squares' slots that no CTA wrote.
__global__ void k_sym_finish(const unsigned long long* __restrict__ sums, int64_t n, double scale, const float* __restrict__ left,
                             float* __restrict__ q, double* __restrict__ sq, int ctas, const int* __restrict__ perm) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t i = perm ? perm[p] : p;
    q[i] = (float)((double)(long long)sums[p] * (left ? scale * (double)left[i] : scale));
    if (sq && p >= ctas) sq[p] = 0.0;
}

template <bool SQ, bool WEIGHTED>
fd_status launch_one(fd_ctx* c, const CUtensorMap& mr, const CUtensorMap& mc, const SymParams& p, int grid) {
    const int smem = smem_total(p.K16);
    // the attribute is per device: set it on every launch (cheap) rather than remembering one device
    // (notes are taken by the pass with squares only)
    const auto kernel = p.near_sums ? (p.list ? k_sym<SQ, WEIGHTED, true, SQ> : k_sym<SQ, WEIGHTED, false, SQ>)
                                    : (p.list ? k_sym<SQ, WEIGHTED, true, false> : k_sym<SQ, WEIGHTED, false, false>);
    FD_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    cudaFuncAttributes fa;
    FD_CUDA(c, cudaFuncGetAttributes(&fa, kernel));
    if (fa.numRegs != kRegsLaunch)
        return fail(c, FD_ERR_UNSUPPORTED, "symmetric row-sum kernel compiled with %d registers per thread, %d expected", fa.numRegs, kRegsLaunch);
    kernel<<<grid, kThreadsS, smem, c->stream>>>(mr, mc, p);
    FD_LAUNCH_CHECK(c, "k_sym");
    return FD_OK;
}

}  // namespace

namespace tc {

fd_status launch_sym_rowsum(fd_ctx* c, const CUtensorMap& mr, const CUtensorMap& mc, const float* weights, const float* left, float* q, double* rowsq,
                            const int* perm, bool use_lists, bool note_near) {
    const Layout& L = c->L;
    SymParams p{};
    p.N = L.N; p.np = L.NP; p.K16 = L.K16;
    p.pairs = (int)(L.NP / 256); p.num_jt = (int)(L.NP / 128);     // (padding gives 2^e = 0)
    p.sums = c->at<unsigned long long>(L.symsum);
    p.sq = rowsq; p.weights = weights; p.status = c->at<unsigned int>(L.status);
    // sums are at most NP 2^bias in the kernel's scaled units (weights at most 1): the fixed-point unit keeps them below 2^61
    int lg = 0;
    while (((int64_t)1 << lg) < L.NP) ++lg;
    p.shift = 61 - kBias - lg;
    FD_CUDA(c, cudaMemsetAsync(p.sums, 0, (size_t)L.N * 8, c->stream));
    if (use_lists) {
        p.list = c->at<unsigned short>(L.lists[rowsq ? 1 : 2]);
        p.counts = c->at<unsigned int>(L.list_counts[rowsq ? 1 : 2]);
        p.uoffs = p.counts + 3 * p.pairs + 1;
    }
    if (note_near) {
        const size_t plane = (size_t)p.num_jt * p.num_jt;
        p.near_product = c->at<unsigned char>(L.near);
        p.near_sums = p.near_product + plane;
        FD_CUDA(c, cudaMemsetAsync(p.near_product, 0, 2 * plane, c->stream));
    }
    // (every pair's own two tiles are listed: there are at least two steps per pair)
    const int grid = (int)std::min<long long>(std::min<long long>(c->sm_count, L.N), use_lists ? 2ll * p.pairs : steps_before(p.pairs, p.num_jt));
    if (rowsq) FD_TRY((launch_one<true, false>(c, mr, mc, p, grid)));
    else FD_TRY((launch_one<false, true>(c, mr, mc, p, grid)));
    k_sym_finish<<<(unsigned)ceil_div(L.N, 256), 256, 0, c->stream>>>(p.sums, L.N, std::ldexp(1.0, -(p.shift + kBias)), left, q, rowsq, grid, perm);
    FD_LAUNCH_CHECK(c, "k_sym_finish");
    return FD_OK;
}

}  // namespace tc

}  // namespace fd
