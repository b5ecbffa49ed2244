// PTX wrappers and constants shared by the tensor-core kernels (tcgen05 / TMEM / TMA / mbarrier, sm_100a).
#pragma once

#include <cuda.h>

#include "fd_internal.h"

namespace fd {
namespace tc {

constexpr int kStages = 4;
constexpr int kThreads = 384;                // row-sum kernel: warps 0-3 / 4-7 exponential warpgroups; warps 8-11: TMA, 2 idle, MMA
constexpr int kBias = 15;                    // P' = 2^15 P keeps fp16 hi/lo of P out of the denormal range (added to the exponent by the Gram MMAs:
                                             // a multiplication after the exponential cost the product at N = 2^20 3 %)
constexpr uint32_t kTmemCols = 512;
constexpr long long kWaitCycles = 4000000000ll;   // ~2 s: far beyond any legitimate wait

struct TcParams {
    int64_t Nrow, N;             // valid rows / columns
    int num_work;                // row-pair tiles (256 rows each)
    int num_jt;                  // column tiles
    int jt_chunk, num_chunks;    // the column range is swept in chunks small enough for L2 (block mode); all CTAs work on one chunk at a time
    int64_t np_rows;             // padded row count of the operand arrays (row index of K slab c = c * np + p)
    int64_t np_cols;
    int K16;
    int b;                       // real block columns to store
    int flush;                   // column tiles per accumulator flush
    const float* left;           // may be null
    const float* colscale_inv;   // per column: 2^-bias / colscale
    float* Y; int64_t ldy;       // block products: output block
    float* q; double* rowsq;     // row-sum modes: outputs
    const float* weights;        // row-sum modes without squares: right weights, padded with zeros to whole tiles
    const int* perm;             // row of Y, q and left for each row of the operand (null: the same)
    int ordered;                 // the columns are in the points' order
    int use_lists;               // block product: the tile lists of the context hold for this pass
    unsigned int* status;
};

// ------------------------------------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Index of this warp in a register the compiler knows to be the same for the whole warp.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
// True in one thread of a converged warp.  The issuing roles run under this and not under `lane == 0`: with elect.sync the
// compiler keeps descriptors and addresses in uniform registers, where tcgen05.mma and TMA read them; under a lane test it
// moves every operand of every instruction there first, and an MMA then costs about 45 SM clocks whatever its width.
// Measured for back-to-back M128 K16, A in TMEM, N = 16 / 32 / 64: 9 / 16 / 32 clocks (the math rate) against 45 / 45 / 45.
// The fp32-grade product at N = 2^20, b = 64 went from 521 to 473 ms with it, N = 2^17, b = 32 from 7.30 to 5.91 ms.
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: returns false (and raises the abort flag) when the limit is hit or another role aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, unsigned int* status, int code,
                                          long long limit = kWaitCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        __nanosleep(40);            // back off: many warps polling shared memory slow the MMA issuer down
        if ((++spins & 63) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit) {
                *abort_flag = 1;
                atomicCAS(status, 0u, (unsigned)(0x100 | code));
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(smem_dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

// Lean issue forms: the 64-bit shared-memory descriptor is passed as (low word, high word), so that stepping through an
// operand costs one 32-bit add on the low word (start-address field, 16-byte units; it cannot carry out of its 14 bits for
// any address below 256 KB), and `accumulate` is a compile-time constant.  The issuing thread shares its scheduler with busy
// warps, so every instruction it does not have to issue shortens the gap between two MMAs.
template <int ACC>
__device__ __forceinline__ void mma_ts2(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 bd;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 bd, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], bd, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(ACC) : "memory");
}
template <int ACC>
__device__ __forceinline__ void mma_ss2(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 ad, bd;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 ad, {%1, %2};\n\tmov.b64 bd, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], ad, bd, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(ACC) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t addr, const uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
        ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 2^x for two values on the FMA pipe: Cody-Waite reduction (W. J. Cody, W. Waite, Software Manual for the Elementary Functions, 1980) to
// x = n + f with |f| <= 1/2, 2^f = 1 + f q(f) with q fitted for the least maximum of the relative error (2e-9; with the rounding of fp32 at most
// 8e-8, 2.7e-8 on average: less than the MUFU's 2^-22), n added to the exponent.  Below 2^-126: 2^-126.  Thirteen instructions for two values
// where the MUFU takes sixteen clocks of its pipe: for kernels that have issue slots to spare.
__device__ __forceinline__ float2 ex2_fma2(float x0, float x1) {
    constexpr float kRound = 12582912.0f;                     // 1.5 2^23: adding it rounds to an integer in the low mantissa bits
    const uint64_t x = pair2(fmaxf(x0, -126.0f), fmaxf(x1, -126.0f));
    const uint64_t t = add2(x, pair2(kRound, kRound));
    const uint64_t f = sub2(x, add2(t, pair2(-kRound, -kRound)));
    uint64_t q = pair2(0.00015353363f, 0.00015353363f);
    q = fma2(q, f, pair2(0.0013398875f, 0.0013398875f));
    q = fma2(q, f, pair2(0.009618437f, 0.009618437f));
    q = fma2(q, f, pair2(0.055503324f, 0.055503324f));
    q = fma2(q, f, pair2(0.24022648f, 0.24022648f));
    q = fma2(q, f, pair2(0.6931472f, 0.6931472f));
    q = fma2(q, f, pair2(1.0f, 1.0f));
    const float2 qs = split2(q), ts = split2(t);
    return make_float2(__int_as_float(__float_as_int(qs.x) + (__float_as_int(ts.x) << 23)), __int_as_float(__float_as_int(qs.y) + (__float_as_int(ts.y) << 23)));
}
__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// h - x for the low / high half h of a packed pair of fp16 values and an fp32 x: one instruction (the conversion of h alone takes two and a half).
__device__ __forceinline__ float sub_lo_f16(uint32_t h, float x) {
    float d;
    asm("{\n\t.reg .b16 l, u;\n\tmov.b32 {l, u}, %1;\n\tsub.f32.f16 %0, l, %2;\n\t}" : "=f"(d) : "r"(h), "f"(x));
    return d;
}
__device__ __forceinline__ float sub_hi_f16(uint32_t h, float x) {
    float d;
    asm("{\n\t.reg .b16 l, u;\n\tmov.b32 {l, u}, %1;\n\tsub.f32.f16 %0, u, %2;\n\t}" : "=f"(d) : "r"(h), "f"(x));
    return d;
}
// K-major shared-memory operand descriptor (sm_100 format): start address, stride between 8-row groups,
// swizzle mode (2 = 128 B rows, 4 = 64 B rows).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t sbo_bytes, uint32_t layout) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(sbo_bytes >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)layout << 61;
    return d;
}
// Instruction descriptor: fp16 x fp16 -> fp32, both operands K-major, M = 128.
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
constexpr uint32_t kNegateA = 1u << 13;      // instruction descriptor: D (+)= -A B

// Reduced-precision block product (fd_tc_fast.cu): one row tile per CTA, work items of 128 rows.
fd_status launch_fast_product(fd_ctx* c, int BT, const CUtensorMap& mr, const CUtensorMap& mc, const CUtensorMap& mh,
                              const TcParams& p, int grid);
// Row sums of the context's whole point set from the tiles on or above the diagonal (fd_tc_sym.cu): q = left * sum_j weights_j K_ij (no
// weights: 1, and the total of rowsq's N entries is sum_ij K_ij^2).
fd_status launch_sym_rowsum(fd_ctx* c, const CUtensorMap& mr, const CUtensorMap& mc, const float* weights, const float* left, float* q,
                            double* rowsq, const int* perm, bool use_lists, bool note_near);
// fp32-grade block product of BT = 16, 32, 48 or 64 columns (fd_tc_block.cu).
fd_status launch_block_product(fd_ctx* c, int BT, const CUtensorMap& mr, const CUtensorMap& mc, const CUtensorMap& mw,
                               const TcParams& tp);

}  // namespace tc
}  // namespace fd
