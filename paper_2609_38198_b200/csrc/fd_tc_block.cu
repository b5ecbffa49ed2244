// fp32-grade block product Y_I += K_IJ W_J on tcgen05 / TMEM (Eqs. 5-6): the kernel behind fd_apply in the fp32-grade mode on
// the Gram-form path.
//
// Per (row tile I, column tile J) of 128 x 128 pairs:
//   1. Gram MMA of augmented fp16 hi|lo points: the tile leaves the tensor core as the base-2 exponent
//        S_ij = 2 b' x_i.x_j - b' r_i - b' r_j + bias      (Eq. 4; the norms ride as extra K columns)
//      into one of three 128-column TMEM buffers.
//   2. Exponential warps (thread = row, 64 columns each) read S, take P = 2^S on the MUFU, split it into fp16 hi (rounded to nearest) and
//      the rest and write both back IN PLACE as the TMEM A operand of the product.  Two values take six instructions: two exponentials, one
//      conversion to a pair of fp16, two mixed-precision subtractions hi - P, one conversion of these; the product MMAs of the
//      second piece negate their A operand.
//   3. Product MMAs per 16-column K step: Y += P_hi W_hi + P_lo W_hi + P_hi W_lo with W = diag(right) V split the same way.
//   4. Every `flush` column tiles a separate warpgroup per row tile adds Y into fp32 registers and the accumulator restarts,
//      so tensor-core accumulation error does not grow with N.
//
// One persistent CTA per SM works on two row tiles (256 rows) at a time, which share each staged column tile; tiles are
// numbered n = 2 j + t (column tile j, row tile t).  28 warps:
//   warps 0-15   exponential warps, four warpgroups: warpgroup k takes column half (k & 1) of row tile (k >> 1);
//   warps 16-23  two flush warpgroups, one per row tile: they own the fp32 accumulator registers and the epilogue;
//   warp 24      TMA producer; warp 25 / 26 product-MMA issuer / Gram-MMA issuer (one elected thread each).
// TMEM (512 columns): three S/P buffers at [0, 384), one accumulator of 64 columns per row tile at 384 + 64 t.
//
// What bounds it: at N >= 2^17 the board's power limit (1000 W), below that the chain of steps that a buffer goes through: 1260 SM clocks a tile at
// N = 50021, b = 20, where the MUFU needs 1024.  Without the exponentials (a probe) the chain still takes 1105, without the product MMAs
// 1210, without two of the three Gram MMAs 1245; exponentials moved to the FMA pipe (a polynomial for one or two columns in sixteen) cost 4 to 10 %.
// Instructions count twice, as issue slots in the chain and as power: hi cut from the bits and subtracted (eight instructions for two values) and
// scalar flushes took 798 instead of 749 us there, 5.45 instead of 5.19 ms at N = 2^17, b = 32, 26.7 instead of 25.6 ms at N = 2^18, b = 64.  Sixteen exponential warps and a product issued per 32-column quarter keep the chain exponentials -> product ->
// Gram -> exponentials of a buffer shorter than the other row tile's exponentials.  Per tile: 1024 SM clocks of MUFU, 193 K16 clocks of Gram MMAs, 12 BT clocks of product MMAs.  Up to 32 columns
// the W_lo product shares an instruction with the W_hi one (B operand [W_hi | W_lo], N = 2 BT) and P_lo W_hi is added to
// the W_lo half of the accumulator: 16 MMAs a tile instead of 24, and the sum of the large terms sees 8 round-toward-zero additions
// per tile instead of 24 (scale error of K V beyond the exponents' own with a flush every tile: 1.5e-7 / 1.2e-7 for positive /
// random-sign V against 1.5e-7 / 5.4e-7 with three terms in one accumulator; a flush every two tiles is 2 % faster and doubles it).
// Measured against the layout it replaced (8 exponential warps that also owned the accumulators, three separate terms, whole
// row pairs per CTA with half-range items for the last round), with the same elected issue: N = 2^20, b = 64: 473 -> 429 ms;
// N = 2^17, b = 32: 5.91 -> 5.31 ms; N = 2^18, D = 30, b = 32: 28.5 -> 26.5 ms; N = 50021, b = 20: 1.03 -> 0.81 ms.
//
// Work is a flat sequence of (row pair, column tile) steps cut into equal ranges, one per CTA, so no size leaves the last round
// of CTAs partly filled.  A row pair that a cut falls into is finished by k_block_fix: every CTA leaves its share in a slot
// of its own and the shares are added in the order of the CTAs, so results do not depend on timing.
#include <algorithm>

#include "fd_tc_common.h"

namespace fd {

namespace {

using namespace tc;

constexpr int kSumFlushes = 32;    // flushes per register sum where the points are ordered
constexpr int kThreadsB = 896;
constexpr int kRegsLaunch = 72, kRegsExp = 72, kRegsFlush = 88, kRegsUtil = 40;
static_assert(kThreadsB * kRegsLaunch == 512 * kRegsExp + 256 * kRegsFlush + 128 * kRegsUtil,
              "setmaxnreg must conserve the register total");

template <int BT>
struct SmemB {
    static constexpr int kXChunk = 128 * 64;                          // one K slab (hi|lo) of 128 points: 8 KB
    static constexpr int kWPart = BT * 128;                           // 64 j x BT columns fp16
    static constexpr int kWBytes = 4 * kWPart;                        // [j-half 0: W_hi, W_lo][j-half 1: W_hi, W_lo]
    static __host__ __device__ constexpr int stage_bytes(int K16) { return K16 * kXChunk + kWBytes; }
    static __host__ __device__ constexpr int total(int K16, int stages) {
        return 1024 /*align slack*/ + stages * stage_bytes(K16) + 2 * K16 * kXChunk + 1024 /*barriers*/;
    }
};

struct BarriersB {
    uint64_t full[kStages], empty[kStages];   // column stage: TMA -> issuers; product issuer -> TMA
    uint64_t xfull, xempty;                   // row operand tiles of a work item
    uint64_t s_full[6];                       // [tile index mod 6]: exponent tile ready (Gram issuer -> one pair of warpgroups)
    uint64_t p_done[3][4];                    // [S buffer][32-column quarter]: P written in place (4 warps -> product issuer)
    uint64_t kw_done[3];                      // [S buffer]: product MMAs that read it have completed (-> Gram issuer)
    uint64_t y_full[2], y_empty[2];           // [row tile]: accumulator flush hand-off (product issuer <-> flush warpgroup)
    uint32_t tmem_base;
    int abort_flag;
};

struct BlockParams {
    int64_t Nrow;
    int64_t np;                  // padded row count of the operand arrays (row index of K slab c = c * np + p)
    int64_t ldy;
    float* Y;
    float* part;                 // slots of [BT][256] floats: two per CTA for shares of row pairs that are cut, then one per CTA for its sums
    const float* left;           // may be null
    const float* colscale_inv;   // per column: 2^-bias / colscale
    unsigned int* status;
    int pairs;                   // row pairs
    int jt0, num_jt;             // column tiles [jt0, jt0 + num_jt) of this launch
    int K16, b, flush, stages;
    int accumulate;              // add to Y (later column chunks) instead of storing
    // tile lists (null: every column tile): column tiles of row pair r at list[r * tiles ..], steps before it offs[r]
    const unsigned short* list; const unsigned int* offs;
    int tiles;
    const int* perm;             // row of Y and left for each row of the operand (null: the same)
};

// First step of CTA `cta` in the flat sequence of steps, and the work item (part of one row pair) that starts at step g of it.
__host__ __device__ __forceinline__ long long range_begin(long long total, int cta, int ctas) { return total * cta / ctas; }
// (a range without steps would leave its slots as they were: no more ranges than steps)
__host__ __device__ __forceinline__ int range_count(long long total, int ctas) { return total < ctas ? (int)total : ctas; }
struct Item { int pair, j0, n; bool whole; };
// Row pair that holds step g of the lists.
__device__ __forceinline__ int pair_of(const BlockParams& p, unsigned int g) {
    int lo = 0, hi = p.pairs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.offs[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
template <bool ORD>
struct Steps {                   // walks a CTA's range item by item
    int pair, j0, left;
    __device__ __forceinline__ Steps(const BlockParams& p) {
        const bool listed = ORD && p.list;
        const long long total = listed ? (long long)p.offs[p.pairs] : (long long)p.pairs * p.num_jt;
        const int ctas = range_count(total, (int)gridDim.x), cta = (int)blockIdx.x;
        if (cta >= ctas) { pair = j0 = left = 0; return; }
        const long long g0 = range_begin(total, cta, ctas);
        pair = listed ? pair_of(p, (unsigned int)g0) : (int)(g0 / p.num_jt);
        j0 = (int)(g0 - (listed ? (long long)p.offs[pair] : (long long)pair * p.num_jt));
        left = (int)(range_begin(total, cta + 1, ctas) - g0);
    }
    __device__ __forceinline__ bool next(const BlockParams& p, Item& it) {
        if (left <= 0) return false;
        const int full = ORD && p.list ? (int)(p.offs[pair + 1] - p.offs[pair]) : p.num_jt;
        it.pair = pair; it.j0 = j0;
        it.n = full - j0 < left ? full - j0 : left;
        it.whole = it.n == full;
        left -= it.n; j0 = 0; ++pair;
        return true;
    }
};

// ORD: the points are ordered (perm, where the rows are the context's own) and tiles may be listed.
template <int BT, bool ORD>
__global__ void __launch_bounds__(kThreadsB, 1)
k_block(const __grid_constant__ CUtensorMap map_xrow, const __grid_constant__ CUtensorMap map_xcol,
        const __grid_constant__ CUtensorMap map_w, const BlockParams p) {
    extern __shared__ uint8_t smem_raw[];
    using SM = SmemB<BT>;
    constexpr bool kConcat = BT <= 32;                 // accumulator [P_hi W_hi | P_hi W_lo + P_lo W_hi], else one sum of three terms
    constexpr uint32_t kYCol = 384;                    // accumulator of row tile t: columns 384 + 64 t ..
    const int K16 = p.K16, stages = p.stages;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_base = base;
    uint8_t* xi_base = base + stages * SM::stage_bytes(K16);                  // 2 row tiles x K16 slabs
    BarriersB* bars = (BarriersB*)(xi_base + 2 * K16 * SM::kXChunk);
    volatile int* abort_flag = &bars->abort_flag;

    const int warp = warp_index(), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
        mbar_init(&bars->xfull, 1); mbar_init(&bars->xempty, 1);
        for (int u = 0; u < 6; ++u) mbar_init(&bars->s_full[u], 1);
        for (int u = 0; u < 3; ++u) {
            mbar_init(&bars->kw_done[u], 1);
            for (int q = 0; q < 4; ++q) mbar_init(&bars->p_done[u][q], 4);
        }
        for (int t = 0; t < 2; ++t) { mbar_init(&bars->y_full[t], 1); mbar_init(&bars->y_empty[t], 4); }
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 24) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    grid_wait();
    grid_go();
    const long long t_begin = clock64();

    if (warp >= 24) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsUtil));
      if (warp == 24) {
        // =============================================================== TMA producer (one thread)
        if (elect_one()) {
            prefetch_tmap(&map_xrow); prefetch_tmap(&map_xcol); prefetch_tmap(&map_w);
            uint32_t issued = 0, s = 0, ph = 1, xph = 1;           // stage ring position and the parity of its "empty" phase
            bool ok = true;
            Steps<ORD> steps(p);
            for (Item it; ok && steps.next(p, it);) {
                ok = mbar_wait(&bars->xempty, xph, abort_flag, p.status, 1);
                if (!ok) break;
                xph ^= 1u;
                mbar_expect_tx(&bars->xfull, 2 * K16 * SM::kXChunk);
                for (int t = 0; t < 2; ++t)
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(xi_base + (t * K16 + c) * SM::kXChunk, &map_xrow, 0,
                                    (int)(c * p.np + (int64_t)it.pair * 256 + t * 128), &bars->xfull);
                for (int j = 0; j < it.n; ++j) {
                    ok = mbar_wait(&bars->empty[s], ph, abort_flag, p.status, 2);
                    if (!ok) break;
                    uint8_t* st = stage_base + s * SM::stage_bytes(K16);
                    const int x0 = (ORD && p.list ? (int)p.list[(size_t)it.pair * p.tiles + it.j0 + j] : p.jt0 + it.j0 + j) * 128;
                    mbar_expect_tx(&bars->full[s], SM::stage_bytes(K16));
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(st + c * SM::kXChunk, &map_xcol, 0, (int)(c * p.np + x0), &bars->full[s]);
                    uint8_t* wst = st + K16 * SM::kXChunk;
                    tma_load_2d(wst, &map_w, x0, 0, &bars->full[s]);
                    tma_load_2d(wst + 2 * SM::kWPart, &map_w, x0 + 64, 0, &bars->full[s]);
                    ++issued;
                    if (++s == (uint32_t)stages) { s = 0; ph ^= 1u; }
                }
            }
            if (!ok) {
                // aborted: let the copies already in flight land before the CTA exits (bounded)
                for (uint32_t k = (issued > (uint32_t)stages ? issued - stages : 0); k < issued; ++k) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(&bars->full[k % stages], (k / stages) & 1) && clock64() - t0 < 20000000ll) {}
                }
            }
        }
      } else if (warp == 26) {
        // =============================================================== Gram MMA issuer (one thread)
        // S(n) = A_t B_j^T as soon as its buffer is free again (the product MMAs of tile n - 3 have completed).
        if (elect_one()) {
            constexpr uint32_t idesc_g = idesc_f16(128);
            const uint64_t xd = smem_desc(smem_u32(xi_base), 512, 4);      // 64 B rows (SWIZZLE_64B), 512 B between 8-row groups
            const uint32_t xi_lo = (uint32_t)xd, xdesc_hi = (uint32_t)(xd >> 32);
            const uint32_t stage_lo = (uint32_t)smem_desc(smem_u32(stage_base), 512, 4);
            const uint32_t stage_step = (uint32_t)(SM::stage_bytes(K16) >> 4);
            constexpr uint32_t kSlab = SM::kXChunk >> 4;
            uint32_t s = 0, sph = 0, slot = 0, kph = 1, six = 0, xph = 0;
            bool ok = true;
            Steps<ORD> steps(p);
            for (Item it; ok && steps.next(p, it);) {
                ok = mbar_wait(&bars->xfull, xph, abort_flag, p.status, 3);
                if (!ok) break;
                xph ^= 1u;
                for (int n = 0; n < 2 * it.n && ok; ++n) {
                    const uint32_t t = (uint32_t)n & 1u;
                    // (first use of a buffer: the phase before the first one counts as complete)
                    ok = mbar_wait(&bars->kw_done[slot], kph, abort_flag, p.status, 5);
                    if (!ok) break;
                    if (t == 0) {
                        ok = mbar_wait(&bars->full[s], sph, abort_flag, p.status, 4);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    // The two small cross terms (hi x lo) go first and the large hi x hi term last: each MMA rounds its
                    // result at the magnitude of its largest addend, so only the final one rounds at full magnitude.
                    const uint32_t s_addr = tmem + 128u * slot;
                    const uint32_t a0 = xi_lo + t * (uint32_t)K16 * kSlab, b0 = stage_lo + s * stage_step;
                    for (int c = 0; c < K16; ++c) {
                        const uint32_t a = a0 + (uint32_t)c * kSlab, b = b0 + (uint32_t)c * kSlab;
                        if (c == 0) mma_ss2<0>(s_addr, a, xdesc_hi, b + 2, xdesc_hi, idesc_g);      // + 2: the lo half starts 32 B into the row
                        else mma_ss2<1>(s_addr, a, xdesc_hi, b + 2, xdesc_hi, idesc_g);
                        mma_ss2<1>(s_addr, a + 2, xdesc_hi, b, xdesc_hi, idesc_g);
                    }
                    for (int c = 0; c < K16; ++c)
                        mma_ss2<1>(s_addr, a0 + (uint32_t)c * kSlab, xdesc_hi, b0 + (uint32_t)c * kSlab, xdesc_hi, idesc_g);
                    tc_commit(&bars->s_full[six]);
                    if (t == 1) { if (++s == (uint32_t)stages) { s = 0; sph ^= 1u; } }
                    if (++slot == 3) { slot = 0; kph ^= 1u; }
                    if (++six == 6) six = 0;
                }
                if (ok) tc_commit(&bars->xempty);                  // the row operand tiles may be replaced
            }
        }
      } else if (warp == 25) {
        // =============================================================== product MMA issuer (one thread)
        if (elect_one()) {
            constexpr uint32_t idesc_hi = idesc_f16(kConcat ? 2 * BT : BT), idesc_lo = idesc_f16(BT), idesc_res = idesc_lo | kNegateA;
            // W stage descriptor as (low, high) words: 128 B rows (SWIZZLE_128B), 1024 B between 8-row groups
            const uint64_t wd = smem_desc(smem_u32(stage_base + K16 * SM::kXChunk), 1024, 2);
            const uint32_t wbase_lo = (uint32_t)wd, wdesc_hi = (uint32_t)(wd >> 32);
            const uint32_t stage_step = (uint32_t)(SM::stage_bytes(K16) >> 4);
            uint32_t s = 0, slot = 0, pph = 0, yph = 1;            // ring positions; yph: parity of the accumulators' "empty" phase
            bool ok = true;
            Steps<ORD> steps(p);
            for (Item it; ok && steps.next(p, it);) {
                int in_group = 0;                                  // column tiles accumulated in the current group
                for (int j = 0; j < it.n && ok; ++j) {
                    const bool group_start = in_group == 0;
                    const bool group_end = in_group + 1 == p.flush || j + 1 == it.n;
                    in_group = group_end ? 0 : in_group + 1;
                    const uint32_t w_lo = wbase_lo + s * stage_step;
                    for (uint32_t t = 0; t < 2 && ok; ++t) {
                        const uint32_t p_addr = tmem + 128u * slot, y_addr = tmem + kYCol + 64u * t;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            // the two warpgroups of a row tile finish their first quarters (0, 2) first
                            const int q = ((i & 1) << 1) | (i >> 1);
                            ok = mbar_wait(&bars->p_done[slot][q], pph, abort_flag, p.status, 7);
                            if (!ok) break;
                            if (i == 0 && group_start) {
                                // (first group: the "empty" phase before the first one counts as complete)
                                ok = mbar_wait(&bars->y_empty[t], yph, abort_flag, p.status, 6);
                                if (!ok) break;
                            }
                            tc_fence_after();
                            // K step k of quarter q: P_hi at S-buffer columns 32 q + [16 k, 16 k + 8), P_lo in the next eight; W rows of
                            // the quarter's j-half start 32 B (two 16-byte units) further per K step
                            const uint32_t bq = w_lo + (uint32_t)(((q >> 1) * 2 * SM::kWPart) >> 4) + 4u * (q & 1);
                            const uint32_t aq = p_addr + 32u * q;
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                if constexpr (kConcat) {
                                    if (k == 0 && i == 0 && group_start) mma_ts2<0>(y_addr, aq, bq, wdesc_hi, idesc_hi);
                                    else mma_ts2<1>(y_addr, aq + 16 * k, bq + 2 * k, wdesc_hi, idesc_hi);
                                    mma_ts2<1>(y_addr + BT, aq + 16 * k + 8, bq + 2 * k, wdesc_hi, idesc_res);
                                } else {
                                    // the two small terms of both K steps first: what they round away is smaller then
                                    if (k == 0 && i == 0 && group_start) mma_ts2<0>(y_addr, aq + 8, bq, wdesc_hi, idesc_res);
                                    else mma_ts2<1>(y_addr, aq + 16 * k + 8, bq + 2 * k, wdesc_hi, idesc_res);
                                    mma_ts2<1>(y_addr, aq + 16 * k, bq + (uint32_t)(SM::kWPart >> 4) + 2 * k, wdesc_hi, idesc_lo);
                                }
                            }
                            if constexpr (!kConcat) {
#pragma unroll
                                for (int k = 0; k < 2; ++k) mma_ts2<1>(y_addr, aq + 16 * k, bq + 2 * k, wdesc_hi, idesc_lo);
                            }
                        }
                        if (!ok) break;
                        tc_commit(&bars->kw_done[slot]);
                        if (group_end) tc_commit(&bars->y_full[t]);
                        if (++slot == 3) { slot = 0; pph ^= 1u; }
                    }
                    if (!ok) break;
                    if (group_start) yph ^= 1u;
                    tc_commit(&bars->empty[s]);
                    if (++s == (uint32_t)stages) s = 0;
                }
            }
        }
      }
    } else if (warp >= 16) {
        // =============================================================== flush warpgroup of row tile t (thread = row)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsFlush));
        const int t = (warp - 16) >> 2;
        const int wq = warp & 3;                       // TMEM lane quarter this warp may access
        const uint32_t y_addr = tmem + ((uint32_t)(wq * 32) << 16) + kYCol + 64u * t;
        const int row_in_pair = t * 128 + wq * 32 + lane;
        uint32_t yph = 0;
        bool ok = true;
        Steps<ORD> steps(p);
        for (Item it; ok && steps.next(p, it);) {
            uint64_t acc2[BT / 2];
#pragma unroll
            for (int c = 0; c < BT / 2; ++c) acc2[c] = 0;
            // The tensor core adds each K step into the TMEM accumulator with round-toward-zero.  For a sum whose partial sums
            // keep one sign, n additions lose n / 4 ulp of the result on average (half an ulp each, at a running magnitude that
            // averages half the final one): 2^-25 of the result per addition.  The flush adds that expected loss back.  (With
            // the small terms in columns of their own only the 8 large additions per tile count.)
            // Two-level sums where the points are ordered: every kSumFlushes groups the registers go to a slot in memory
            // and restart.  A single fp32 sum over thousands of tiles drops what lies below half a unit in its last place: with ordered
            // points most of the far tiles' shares (N = 2^17, 6-torus: -8.5e-7 of a row's sum, always of the same sign).  In the
            // caller's order the tiles' shares are of one size and the single sum loses nothing of one sign.
            const int period = kSumFlushes * p.flush;
            int left_tiles = it.n;
            while (left_tiles > 0) {
                if constexpr (ORD) {
                    const int done = it.n - left_tiles;
                    if (done > 0 && done % period == 0) {
                        float* sums = p.part + (size_t)(2 * gridDim.x + blockIdx.x) * BT * 256 + row_in_pair;
#pragma unroll
                        for (int c = 0; c < BT; ++c) {
                            const float2 a = split2(acc2[c / 2]);
                            const float v = c & 1 ? a.y : a.x;
                            sums[c * 256] = done == period ? v : sums[c * 256] + v;
                            if (c & 1) acc2[c / 2] = 0;
                        }
                    }
                }
                const int tiles_in_group = left_tiles < p.flush ? left_tiles : p.flush;
                left_tiles -= tiles_in_group;
                const float corr1 = 1.0f + (float)(tiles_in_group * (kConcat ? 8 : 24)) * 2.98023224e-8f;
                const uint64_t corr = pair2(corr1, corr1);
                ok = mbar_wait(&bars->y_full[t], yph, abort_flag, p.status, 10);
                if (!ok) break;
                yph ^= 1u;
                tc_fence_after();
                constexpr int kStep = BT <= 32 ? 16 : 8;           // columns per TMEM load (registers)
#pragma unroll
                for (int c0 = 0; c0 < BT; c0 += kStep) {
                    uint32_t hi[kStep], lo[kStep];
                    if constexpr (kConcat) { tmem_ld16(y_addr + c0, hi); tmem_ld16(y_addr + BT + c0, lo); }
                    else tmem_ld8(y_addr + c0, hi);
                    tmem_wait_ld();
                    if (c0 + kStep == BT) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars->y_empty[t]);
                    }
#pragma unroll
                    for (int c = 0; c < kStep; c += 2) {
                        const uint64_t h2 = pair2(__uint_as_float(hi[c]), __uint_as_float(hi[c + 1]));
                        uint64_t& a2 = acc2[(c0 + c) / 2];
                        if constexpr (kConcat) a2 = add2(a2, fma2(h2, corr, pair2(__uint_as_float(lo[c]), __uint_as_float(lo[c + 1]))));
                        else a2 = fma2(h2, corr, a2);
                    }
                }
            }
            if (!ok) break;
            float acc[BT];
#pragma unroll
            for (int c = 0; c < BT; c += 2) { const float2 a = split2(acc2[c / 2]); acc[c] = a.x; acc[c + 1] = a.y; }
            if constexpr (ORD)
                if (it.n > period) {
                    const float* sums = p.part + (size_t)(2 * gridDim.x + blockIdx.x) * BT * 256 + row_in_pair;
#pragma unroll
                    for (int c = 0; c < BT; ++c) acc[c] += sums[c * 256];
                }
            if (!it.whole) {
                // a share of a row pair that a cut falls into: at most two per CTA (one that starts its row pair, one that does not)
                float* o = p.part + (size_t)(2 * blockIdx.x + (it.j0 == 0 ? 1 : 0)) * BT * 256 + row_in_pair;
#pragma unroll
                for (int c = 0; c < BT; ++c)
                    if (c < p.b) o[c * 256] = acc[c];
                continue;
            }
            int64_t row = (int64_t)it.pair * 256 + row_in_pair;
            if (row < p.Nrow) {
                if (ORD && p.perm) row = p.perm[row];
                const float l = p.left ? p.left[row] : 1.0f;
#pragma unroll
                for (int c = 0; c < BT; ++c)
                    if (c < p.b) {
                        float* o = p.Y + row + (int64_t)c * p.ldy;
                        const float v = acc[c] * l * p.colscale_inv[c];
                        // streaming: the partial results are touched once per column chunk and should not push the operands,
                        // which every CTA re-reads, out of L2
                        __stcs(o, p.accumulate ? __ldcs(o) + v : v);
                    }
            }
        }
    } else {
        // =============================================================== exponential warps
        const int wg = warp >> 2;                      // warpgroup 0..3
        const int t = wg >> 1;                         // row tile it serves
        const int h = wg & 1;                          // column half of every tile it takes
        const int wq = warp & 3;                       // TMEM lane quarter this warp may access
        const uint32_t lane_addr = ((uint32_t)(wq * 32) << 16) + 64u * h;
        uint32_t slot = (uint32_t)t, six = (uint32_t)t, ph = 0;       // tile index mod 3, mod 6, and the phase of s_full[six]
        bool ok = true;
        Steps<ORD> steps(p);
        for (Item it; ok && steps.next(p, it);) {
            for (int j = 0; j < it.n; ++j) {
                ok = mbar_wait(&bars->s_full[six], ph, abort_flag, p.status, 9);
                if (!ok) break;
                tc_fence_after();
                const uint32_t addr = tmem + lane_addr + 128u * slot;
#pragma unroll
                for (int q32 = 0; q32 < 2; ++q32) {
                    uint32_t sv[32];
                    tmem_ld32(addr + 32 * q32, sv);
                    tmem_wait_ld();
#pragma unroll
                    for (int ch = 0; ch < 2; ++ch) {
                        uint32_t hi[8], lo[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float p0 = ex2f(__uint_as_float(sv[16 * ch + 2 * i]));
                            const float p1 = ex2f(__uint_as_float(sv[16 * ch + 2 * i + 1]));
                            hi[i] = pack_f16x2(p0, p1);
                            lo[i] = pack_f16x2(sub_lo_f16(hi[i], p0), sub_hi_f16(hi[i], p1));
                        }
                        tmem_st8(addr + 32 * q32 + 16 * ch, hi);
                        tmem_st8(addr + 32 * q32 + 16 * ch + 8, lo);
                    }
                    // the product of a quarter starts while the next one is still being exponentiated
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->p_done[slot][2 * h + q32]);
                }
                slot += 2; if (slot >= 3) slot -= 3;
                six += 2; if (six >= 6) { six -= 6; ph ^= 1u; }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    // SM cycles CTA 0 spent on its work items (status words 2-3): lets the host relate the kernel time to the SM clock
    // (a product in several column chunks adds its launches up)
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        long long* cycles = reinterpret_cast<long long*>(p.status + 2);
        *cycles = clock64() - t_begin + (p.accumulate ? *cycles : 0);
    }
    if (warp == 24) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Finishes the row pairs that a cut falls into: adds the CTAs' shares in the order of the CTAs.  Block = (row pair, 8 columns).  A product of few rows is
// cut into up to 37 shares a pair: eight are read ahead of their additions (one after the other, with a 64-bit division each: 50 us of
// the 100 of a product of 1000 rows, 16384 points and 16 columns; 26 of 74 so).
template <int BT>
__global__ void __launch_bounds__(256)
k_block_fix(const BlockParams p, int ctas) {
    grid_wait();
    grid_go();
    const int pair = blockIdx.x;
    const long long total = p.list ? (long long)p.offs[p.pairs] : (long long)p.pairs * p.num_jt;
    const long long g0 = p.list ? (long long)p.offs[pair] : (long long)pair * p.num_jt;
    const long long g1 = p.list ? (long long)p.offs[pair + 1] : g0 + p.num_jt;
    ctas = range_count(total, ctas);
    // the last CTA whose range begins at or before step g0, and the last one whose range begins before g1
    const int first = (int)(((g0 + 1) * ctas - 1) / total), last = (int)((g1 * ctas - 1) / total);
    if (first == last) return;                                         // not cut: the CTA stored it
    int64_t row = (int64_t)pair * 256 + threadIdx.x;
    if (row >= p.Nrow) return;
    if (p.perm) row = p.perm[row];
    const int c0 = (int)blockIdx.y * 8;
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.f;
#pragma unroll 8
    for (int cta = first; cta <= last; ++cta) {
        // the share whose item starts the row pair sits in slot 1 of its CTA, every later one in slot 0
        const float* o = p.part + (size_t)(2 * cta + (cta == first ? 1 : 0)) * BT * 256 + threadIdx.x;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c0 + c < p.b) acc[c] += o[(c0 + c) * 256];
    }
    const float l = p.left ? p.left[row] : 1.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c0 + c < p.b) {
            float* o = p.Y + row + (int64_t)(c0 + c) * p.ldy;
            const float v = acc[c] * l * p.colscale_inv[c0 + c];
            *o = p.accumulate ? *o + v : v;
        }
}

template <int BT>
fd_status launch_one(fd_ctx* c, const CUtensorMap& mr, const CUtensorMap& mc, const CUtensorMap& mw, BlockParams p, bool ordered, int jt_total, int jt_chunk) {
    p.stages = kStages;
    while (p.stages > 2 && SmemB<BT>::total(p.K16, p.stages) > 227 * 1024) --p.stages;
    const int smem = SmemB<BT>::total(p.K16, p.stages);
    if (smem > 227 * 1024) return fail(c, FD_ERR_UNSUPPORTED, "block product kernel needs %d B of shared memory", smem);
    // the attribute is per device: set it on every launch (cheap) rather than remembering one device
    const auto kernel = ordered ? k_block<BT, true> : k_block<BT, false>;
    FD_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    cudaFuncAttributes fa;
    FD_CUDA(c, cudaFuncGetAttributes(&fa, kernel));
    if (fa.numRegs != kRegsLaunch)
        return fail(c, FD_ERR_UNSUPPORTED, "block product kernel compiled with %d registers per thread, %d expected", fa.numRegs, kRegsLaunch);
    // (with lists: one launch over everything; consecutive row pairs are neighbours and share most of their column tiles)
    if (p.list) jt_chunk = jt_total;
    for (int j0 = 0; j0 < jt_total; j0 += jt_chunk) {
        p.jt0 = j0;
        p.num_jt = std::min(jt_chunk, jt_total - j0);
        p.accumulate = j0 > 0;
        // (with lists the number of steps is known to the device only)
        const long long total = (long long)p.pairs * p.num_jt;
        const int grid = (int)std::min<long long>(c->sm_count, total);
        if ((size_t)3 * grid * BT * 256 > c->L.part_floats) return fail(c, FD_ERR_WORKSPACE, "no room for the shares of cut row pairs");
        FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)grid), dim3(kThreadsB), (size_t)smem, kernel, mr, mc, mw, p));
        FD_LAUNCH_CHECK(c, "k_block");
        bool cut = p.list != nullptr;
        for (int i = 1; i < grid && !cut; ++i) cut = range_begin(total, i, grid) % p.num_jt != 0;
        if (cut) {
            FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)p.pairs, (unsigned)ceil_div(p.b, 8)), dim3(256), 0, k_block_fix<BT>, p, grid));
            FD_LAUNCH_CHECK(c, "k_block_fix");
        }
    }
    return FD_OK;
}

}  // namespace

namespace tc {

// tp: the block product's parameters (Nrow, np_rows, K16, b, flush, left, colscale_inv, Y, ldy, num_work, num_jt, jt_chunk)
fd_status launch_block_product(fd_ctx* c, int BT, const CUtensorMap& mr, const CUtensorMap& mc, const CUtensorMap& mw, const TcParams& tp) {
    BlockParams p{};
    p.Nrow = tp.Nrow; p.np = tp.np_rows; p.ldy = tp.ldy; p.Y = tp.Y; p.left = tp.left; p.colscale_inv = tp.colscale_inv;
    p.status = tp.status; p.part = c->at<float>(c->L.part);
    p.pairs = tp.num_work; p.K16 = tp.K16; p.b = tp.b; p.flush = tp.flush; p.perm = tp.perm;
    if (tp.use_lists) {
        p.list = c->at<unsigned short>(c->L.lists[0]);
        p.offs = c->at<unsigned int>(c->L.list_counts[0]) + 2 * p.pairs;
        p.tiles = (int)(c->L.NP / 128);
    }
    switch (BT) {
        case 16: return launch_one<16>(c, mr, mc, mw, p, tp.ordered != 0, tp.num_jt, tp.jt_chunk);
        case 32: return launch_one<32>(c, mr, mc, mw, p, tp.ordered != 0, tp.num_jt, tp.jt_chunk);
        case 48: return launch_one<48>(c, mr, mc, mw, p, tp.ordered != 0, tp.num_jt, tp.jt_chunk);
        case 64: return launch_one<64>(c, mr, mc, mw, p, tp.ordered != 0, tp.num_jt, tp.jt_chunk);
    }
    return fail(c, FD_ERR_UNSUPPORTED, "no block product instantiation for column tile %d", BT);
}

}  // namespace tc

}  // namespace fd
