// Gram-form row sums on the 5th-generation tensor cores (tcgen05 + TMEM), Eqs. 4-6, the operand packing and the host side of every
// Gram-form pass.  (The block products' kernels: fd_tc_block.cu, fp32-grade; fd_tc_fast.cu, reduced precision.)
//
// Per (row tile I, column tile J) of 128 x 128 pairs:
//   1. Gram MMA (fp16 hi/lo split, three products per 16-wide K slab, fp32 accumulation in TMEM)
//      of AUGMENTED points, so the tile leaves the tensor core already as the base-2 exponent
//        S_ij = 2 b' x_i.x_j - b' r_i - b' r_j + bias            (b' = beta log2 e, Eq. 4)
//      the norms ride along as extra K columns ([.., e_i, 1] . [.., 1, e_j]), each norm carried by
//      two hi/lo pairs so it is exact to fp32.
//   2. Two warpgroups (one per row tile; thread = row) read S from TMEM, take 2^S on the MUFU and add P (and P^2).
// S tiles flow through a ring of TMEM buffers shared by both row tiles, so the tensor core runs ahead of the warpgroups.
// Rectangular and row-sharded passes: the warpgroups add P (and P^2) on the FMA pipe,
// fp32 within a column tile and fp64 across tiles; a right vector multiplies P.
// (The degree passes of a whole data set use K = K^T: fd_tc_sym.cu.)
//
// One persistent CTA per SM: warps 0-3 / 4-7 = the two exponential warpgroups (raised to 232 registers); warp 8 = TMA producer,
// warp 11 = Gram-MMA issuer (lowered to 40 registers).  Column tiles are staged by TMA (every CTA loads its own copy) through
// a 4-deep ring.  Every mbarrier wait is bounded; on expiry the CTA raises a status word, drains and exits.
#include <cuda.h>

#include <algorithm>
#include <cmath>

#include "fd_tc_common.h"

namespace fd {

namespace {

using namespace tc;

// ------------------------------------------------------------------------------------------------ shared memory map
struct Smem {
    static constexpr int kXChunk = 128 * 64;                       // one K slab (hi|lo) of 128 points: 8 KB
    static __host__ __device__ constexpr int stage_bytes(int K16) { return K16 * kXChunk; }
    static __host__ __device__ constexpr int total(int K16) {
        return 1024 /*align slack*/ + kStages * stage_bytes(K16) + 2 * K16 * kXChunk + 1024 /*barriers*/;
    }
};

constexpr int kMaxBuf = 4;

struct Barriers {
    uint64_t full[kStages], empty[kStages];
    uint64_t xfull, xempty;
    // Ring-buffer barriers are indexed [buffer][row tile]: each one then has a single producer role and a single
    // consumer role that waits on EVERY one of its phases.  (A parity wait is only unambiguous if the waiter has seen
    // the previous phase complete; a barrier per buffer alone, shared by both row tiles, lets a waiter that skips
    // alternate phases pass one phase early.)
    uint64_t s_full[kMaxBuf][2];            // S tile ready in ring buffer (Gram issuer -> warpgroup)
    uint64_t s_done[kMaxBuf][2];            // S consumed (warpgroup -> issuer)
    uint32_t tmem_base;
    int abort_flag;
};

// ------------------------------------------------------------------------------------------------ work items
// Work item w of a CTA: row pair blockIdx.x + w * gridDim.x, all column tiles.

// ------------------------------------------------------------------------------------------------ the kernel
// Tiles of one work item are numbered n = 2 j + t (column tile j, row tile t) and flow through a ring of four S buffers in
// TMEM, so the tensor core runs up to four tiles ahead of the warpgroups.  BT = 16: with the sum of squares, 32: with weights.
template <int BT>
__global__ void __launch_bounds__(kThreads, 1)
k_tc(const __grid_constant__ CUtensorMap map_xrow, const __grid_constant__ CUtensorMap map_xcol, const TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    using SM = Smem;
    constexpr int NBUF = 4;
    constexpr uint32_t kRingPeriod = NBUF;             // tiles between two uses of a buffer by the same row tile
    const int K16 = p.K16;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_base = base;
    uint8_t* xi_base = base + kStages * SM::stage_bytes(K16);                 // 2 row tiles x K16 slabs
    Barriers* bars = (Barriers*)(xi_base + 2 * K16 * SM::kXChunk);
    volatile int* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
        mbar_init(&bars->xfull, 1); mbar_init(&bars->xempty, 1);
        for (int u = 0; u < kMaxBuf; ++u)
            for (int t = 0; t < 2; ++t) {
                mbar_init(&bars->s_full[u][t], 1); mbar_init(&bars->s_done[u][t], 4);
            }
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    const long long t_begin = clock64();

    const int num_jt = p.num_jt, tiles_per_item = 2 * num_jt;
    const int my_items = (p.num_work - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(40));
      if (warp == 8) {
        // =============================================================== TMA producer (one thread)
        if (lane == 0) {
            prefetch_tmap(&map_xrow); prefetch_tmap(&map_xcol);
            uint32_t it = 0;
            bool ok = true;
            for (int w = 0; w < my_items && ok; ++w) {
                const int item = (int)blockIdx.x + w * (int)gridDim.x;
                ok = mbar_wait(&bars->xempty, (w & 1) ^ 1, abort_flag, p.status, 1);
                if (!ok) break;
                mbar_expect_tx(&bars->xfull, 2 * K16 * SM::kXChunk);
                for (int t = 0; t < 2; ++t)
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(xi_base + (t * K16 + c) * SM::kXChunk, &map_xrow, 0,
                                    (int)(c * p.np_rows + (int64_t)item * 256 + t * 128), &bars->xfull);
                for (int j = 0; j < num_jt; ++j, ++it) {
                    const int s = it % kStages;
                    ok = mbar_wait(&bars->empty[s], ((it / kStages) & 1) ^ 1, abort_flag, p.status, 2);
                    if (!ok) break;
                    uint8_t* st = stage_base + s * SM::stage_bytes(K16);
                    mbar_expect_tx(&bars->full[s], SM::stage_bytes(K16));
                    for (int c = 0; c < K16; ++c)
                        tma_load_2d(st + c * SM::kXChunk, &map_xcol, 0, (int)(c * p.np_cols + (int64_t)j * 128), &bars->full[s]);
                }
            }
            if (!ok) {
                // aborted: let the copies already in flight land before the CTA exits (bounded)
                const uint32_t issued = it;
                for (uint32_t k = (issued > (uint32_t)kStages ? issued - kStages : 0); k < issued; ++k) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(&bars->full[k % kStages], (k / kStages) & 1) && clock64() - t0 < 20000000ll) {}
                }
            }
        }
      } else if (warp == 11) {
        // =============================================================== Gram MMA issuer (one thread)
        // Issues S(n) = A_t B_j^T for every tile as soon as its ring buffer is free again; runs up to NBUF tiles ahead.
        if (lane == 0) {
            // The MUFU binds and the tensor pipe is mostly idle; descriptors are rebuilt per MMA under a plain lane test, which paces
            // the Gram MMAs between the warpgroups' TMEM loads (issuing them in tight bursts measured 5 % slower, electing
            // the thread with elect.sync 2 %).
            constexpr uint32_t idesc_g = idesc_f16(128);
            uint32_t it0 = 0, gn0 = 0;
            bool ok = true;
            for (int w = 0; w < my_items && ok; ++w) {
                ok = mbar_wait(&bars->xfull, w & 1, abort_flag, p.status, 3);
                if (!ok) break;
                tc_fence_after();
                for (int n = 0; n < tiles_per_item && ok; ++n) {
                    const uint32_t g = gn0 + (uint32_t)n;
                    const int buf = g % NBUF;
                    const uint32_t itj = it0 + (uint32_t)(n >> 1);
                    const int s = itj % kStages;
                    if (g >= (uint32_t)NBUF) {
                        // the tile that used this buffer last (NBUF tiles ago, possibly of the other row tile) must be finished
                        const uint32_t gp = g - NBUF;
                        uint64_t* fb = &bars->s_done[buf][gp & 1];
                        ok = mbar_wait(fb, (gp / kRingPeriod) & 1, abort_flag, p.status, 5);
                        if (!ok) break;
                    }
                    if ((n & 1) == 0) {
                        ok = mbar_wait(&bars->full[s], (itj / kStages) & 1, abort_flag, p.status, 4);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    // The two small cross terms (hi x lo) go first and the large hi x hi term last: each MMA rounds its
                    // result at the magnitude of its largest addend, so only the final one rounds at full magnitude.
                    const uint32_t s_addr = tmem + 128u * buf;
                    const int t = n & 1;
                    uint8_t* st = stage_base + s * SM::stage_bytes(K16);
                    for (int c = 0; c < K16; ++c) {
                        uint64_t a = smem_desc(smem_u32(xi_base + (t * K16 + c) * SM::kXChunk), 512, 4);
                        uint64_t b = smem_desc(smem_u32(st + c * SM::kXChunk), 512, 4);
                        mma_ss(s_addr, a, b + 2, idesc_g, c > 0);          // + 2: the lo half starts 32 B into the row
                        mma_ss(s_addr, a + 2, b, idesc_g, 1);
                    }
                    for (int c = 0; c < K16; ++c) {
                        uint64_t a = smem_desc(smem_u32(xi_base + (t * K16 + c) * SM::kXChunk), 512, 4);
                        uint64_t b = smem_desc(smem_u32(st + c * SM::kXChunk), 512, 4);
                        mma_ss(s_addr, a, b, idesc_g, 1);
                    }
                    tc_commit(&bars->s_full[buf][n & 1]);
                    if (n & 1) tc_commit(&bars->empty[s]);   // both Gram MMAs of this column tile issued
                }
                if (ok) tc_commit(&bars->xempty);                  // the row operand tiles may be replaced
                it0 += (uint32_t)num_jt;
                gn0 += (uint32_t)tiles_per_item;
            }
        }
      }
    } else {
        // =============================================================== exponential warpgroups
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(232));
        const int t = warp >> 2;                       // row tile of this warpgroup
        const int wq = warp & 3;                       // TMEM lane quarter this warp may access
        const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
        const int row_in_tile = wq * 32 + lane;
        uint32_t gn0 = 0;
        bool ok = true;

        for (int w = 0; w < my_items && ok; ++w) {
            const int item = (int)blockIdx.x + w * (int)gridDim.x;
            int64_t row = (int64_t)item * 256 + t * 128 + row_in_tile;
            {
                double dsum = 0.0, dsq = 0.0;
                for (int j = 0; j < num_jt && ok; ++j) {
                    const uint32_t g = gn0 + 2u * j + t;
                    const int buf = g % NBUF;
                    ok = mbar_wait(&bars->s_full[buf][t], (g / kRingPeriod) & 1, abort_flag, p.status, 8);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t addr = tmem + lane_addr + 128u * buf;
                    const float4* wcol = reinterpret_cast<const float4*>(p.weights) + (int64_t)j * 32;
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, q0 = 0.f, q1 = 0.f;
                    uint32_t sv[4][32];
#pragma unroll
                    for (int qd = 0; qd < 4; ++qd) tmem_ld32(addr + 32 * qd, sv[qd]);
                    tmem_wait_ld();
                    // the buffer can be refilled as soon as its values are in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->s_done[buf][t]);
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const float p0 = ex2f(__uint_as_float(sv[ch][i])), p1 = ex2f(__uint_as_float(sv[ch][i + 1]));
                            const float p2 = ex2f(__uint_as_float(sv[ch][i + 2])), p3 = ex2f(__uint_as_float(sv[ch][i + 3]));
                            if (BT == 32) {                // weights instead of the sum of squares (broadcast reads)
                                const float4 w4 = __ldg(wcol + 8 * ch + i / 4);
                                a0 = fmaf(p0, w4.x, a0); a1 = fmaf(p1, w4.y, a1); a2 = fmaf(p2, w4.z, a2); a3 = fmaf(p3, w4.w, a3);
                            } else {
                                a0 += p0; a1 += p1; a2 += p2; a3 += p3;
                                q0 = fmaf(p0, p0, q0); q1 = fmaf(p1, p1, q1); q0 = fmaf(p2, p2, q0); q1 = fmaf(p3, p3, q1);
                            }
                        }
                    }
                    dsum += (double)((a0 + a1) + (a2 + a3));
                    dsq += (double)(q0 + q1);
                }
                if (ok && row < p.Nrow) {
                    if (p.perm) row = p.perm[row];
                    // undo the 2^bias scaling of P (exact powers of two)
                    constexpr double scale = 1.0 / (double)(1 << kBias);
                    p.q[row] = (float)(p.left ? dsum * (scale * (double)p.left[row]) : dsum * scale);
                    if (p.rowsq) p.rowsq[row] = dsq * (scale * scale);
                }
            }
            gn0 += (uint32_t)tiles_per_item;
        }
    }
    tc_fence_before();
    __syncthreads();
    // SM cycles CTA 0 spent on its work items (status words 2-3): lets the host relate the kernel time to the SM clock
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<long long*>(p.status + 2) = clock64() - t_begin;
    if (warp == 8) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Exercises the bounded-wait path without any fault: one thread waits on a barrier that nothing will ever complete,
// with a short limit; the wait gives up, records its code in the status word and the kernel returns normally.
__global__ void k_wait_selftest(unsigned int* status, long long limit_cycles) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_wait(&bar, 0, &abort_flag, status, 0x7f, limit_cycles);
    }
}

// ------------------------------------------------------------------------------------------------ operand packing
// Augmented fp16 hi|lo operand rows.  role 0 (rows of the product): [c x, e, 1]; role 1 (columns): [c x, 1, e] with
// c = sqrt(2 b'), e = -b' |x - mu|^2 (+ the bias for role 1).
// Layout: slab s (16 augmented columns) of point p at out[(s * np + p) * 32 ..]: 16 hi then 16 lo halves.
// Where as many slabs of 12 coordinates suffice (slab_norms), every slab carries the norm of its own coordinates in its last
// four columns: the partial sum over the slabs is then -b' |difference|^2 of the coordinates so far (plus bias), never larger than the
// final exponent, instead of a dot product of the size of the norms that the last slab takes back.  The tensor core
// rounds each MMA at the magnitude of its sum, so this removes most of the exponent's error for far-out points (R^30, exponents
// up to 60: worst eigenvalue error of 33 pairs 9.7e-7 -> 6.6e-7).  Else coordinates first, the four norm columns after the last one.
// One thread per (point, slab, role): the 64 bytes it writes are contiguous.
struct PackRole { const float* xs; __half* out; int64_t n; const int* perm; };   // n: valid points of this role; perm: point of each position
__global__ void __launch_bounds__(256)
k_pack_points(const PackRole rows, const PackRole cols, int first_role, int DP, int D, int64_t np, const double* __restrict__ mu, double bprime,
              double cs, int slab_norms) {
    const int64_t pidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pidx >= np) return;
    const int s = blockIdx.y, role = first_role + (int)blockIdx.z;
    const PackRole pr = role == 0 ? rows : cols;
    const bool valid = pidx < pr.n;
    const float* x = pr.xs + (valid && pr.perm ? (int64_t)pr.perm[pidx] : pidx) * DP;
    const int c0 = slab_norms ? 12 * s : 16 * s;                  // first coordinate of this slab
    const int norm0 = slab_norms ? 12 : D - c0;                   // first norm column inside the slab (may lie outside it)
    __half hi[16], lo[16];
    double r = 0.0;                                               // norm of this slab's coordinates
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
        hi[kk] = lo[kk] = __float2half(0.0f);
        if (valid && c0 + kk < D && kk < norm0) {
            const double d = (double)x[c0 + kk] - mu[c0 + kk], v = cs * d;
            r += d * d;
            hi[kk] = __double2half(v);
            lo[kk] = __double2half(v - (double)__half2float(hi[kk]));
        }
    }
    if (norm0 < 16 && norm0 > -4) {
        if (!slab_norms) {
            r = 0.0;
            if (valid)
                for (int k = 0; k < D; ++k) { const double d = (double)x[k] - mu[k]; r += d * d; }
        }
        double e = -bprime * r;
        if (role == 1 && (s == 0 || !slab_norms)) e += (double)kBias;
        if (!valid && (s == 0 || !slab_norms)) e = -30000.0;      // padded point: 2^e = 0 (its row / column contributes nothing)
        // norm pieces: two hi/lo pairs carry e to beyond fp32 precision
        const __half e_h1 = __double2half(e);
        const double r1 = e - (double)__half2float(e_h1);
        const __half e_l1 = __double2half(r1);
        const double r2 = r1 - (double)__half2float(e_l1);
        const __half e_h2 = __double2half(r2);
        const __half e_l2 = __double2half(r2 - (double)__half2float(e_h2));
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const int q = kk - norm0;                             // 0, 1: row-norm columns (role 0 carries e, role 1 carries 1); 2, 3: column-norm
            if (q < 0 || q > 3) continue;
            if ((q >> 1) == role) { hi[kk] = (q & 1) ? e_h2 : e_h1; lo[kk] = (q & 1) ? e_l2 : e_l1; }
            else { hi[kk] = __float2half(1.0f); lo[kk] = __float2half(0.0f); }
        }
    }
    uint4* o = reinterpret_cast<uint4*>(pr.out + ((int64_t)s * np + pidx) * 32);
    auto two = [](__half a, __half b) { return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16); };
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        o[q] = make_uint4(two(hi[8 * q], hi[8 * q + 1]), two(hi[8 * q + 2], hi[8 * q + 3]), two(hi[8 * q + 4], hi[8 * q + 5]), two(hi[8 * q + 6], hi[8 * q + 7]));
        o[2 + q] = make_uint4(two(lo[8 * q], lo[8 * q + 1]), two(lo[8 * q + 2], lo[8 * q + 3]), two(lo[8 * q + 4], lo[8 * q + 5]), two(lo[8 * q + 6], lo[8 * q + 7]));
    }
}

// out[j] = w[j] (1 without w) for j < n, 0 up to np: the weights of a row sum, padded to whole column tiles.
__global__ void k_pad_weights(const float* __restrict__ w, int64_t n, int64_t np, const int* __restrict__ perm, float* __restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < np) out[j] = j < n ? (w ? w[perm ? perm[j] : j] : 1.f) : 0.f;
}

// Per-block maxima of |right_j V_jc| for each column c (columns from vcols on are the ones vector); infinite where an entry is not finite.
__global__ void __launch_bounds__(256)
k_colmax_partial(const float* __restrict__ V, int64_t ldv, int vcols, const float* __restrict__ right, int64_t N, int c0, float* __restrict__ part) {
    grid_wait();
    grid_go();
    __shared__ float sm[8];
    const bool ones = c0 + (int)blockIdx.y >= vcols;
    const float* v = V + (int64_t)(ones ? 0 : c0 + blockIdx.y) * ldv;
    float m = 0.f;
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < N; j += (int64_t)gridDim.x * 256) {
        float x = ones ? 1.f : v[j];
        if (right) x *= right[j];
        m = fmaxf(m, isfinite(x) ? fabsf(x) : INFINITY);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 8) {
        m = sm[threadIdx.x];
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffu, m, off));
        if (threadIdx.x == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = m;
    }
}
// wt [c * np + j] = fp16 hi piece of scale_c * right_j * V[j, c0 + c], and the lo piece BT rows below when `with_lo`; zero padding for
// j >= N and c >= bc.  scale_c = the power of two that puts the column maximum in [2^12, 2^13): every block reduces the
// partial maxima of its column itself (they are at most 256 values); the first one stores the epilogue factor 2^-bias / scale.
// An entry that is not finite makes its whole column NaN in the fp32-grade mode (the lo piece of Inf is NaN, and 0 NaN = NaN in every
// row): the factor is NaN then, so that rows whose tiles leave the entry out get it too.
__global__ void __launch_bounds__(256)
k_pack_wt(const float* __restrict__ V, int64_t ldv, int vcols, const float* __restrict__ right, int64_t N, int64_t np, int c0, int bc,
          const float* __restrict__ part, int parts, float* __restrict__ inv, __half* __restrict__ wt, int with_lo, const int* __restrict__ perm) {
    grid_wait();
    grid_go();
    __shared__ float sm[8];
    const int c = blockIdx.y;
    float m = c < bc && (int)threadIdx.x < parts ? part[(size_t)c * parts + threadIdx.x] : 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    m = sm[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) m = fmaxf(m, sm[w]);
    float sc = 1.0f;
    if (m > 0.f && isfinite(m)) {
        int e;
        frexpf(m, &e);                               // m = f * 2^e, f in [0.5, 1)
        sc = ldexpf(1.0f, 13 - e);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) inv[c] = with_lo && isinf(m) ? NAN : ldexpf(1.0f, -kBias) / sc;
    const bool ones = c0 + c >= vcols;
    const float* v = V + (int64_t)(ones ? 0 : c0 + c) * ldv;
    __half2* hi = reinterpret_cast<__half2*>(wt + (int64_t)c * np);
    __half2* lo = reinterpret_cast<__half2*>(wt + (int64_t)(gridDim.y + c) * np);
    for (int64_t j2 = (int64_t)blockIdx.x * 256 + threadIdx.x; j2 < np / 2; j2 += (int64_t)gridDim.x * 256) {
        float x[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t j = 2 * j2 + u;
            x[u] = 0.f;
            if (c < bc && j < N) {
                const int64_t i = perm ? (int64_t)perm[j] : j;
                const float y = ones ? 1.f : v[i];
                x[u] = (right ? y * right[i] : y) * sc;
            }
        }
        const __half2 h = __floats2half2_rn(x[0], x[1]);
        hi[j2] = h;
        if (with_lo) lo[j2] = __floats2half2_rn(x[0] - __low2float(h), x[1] - __high2float(h));
    }
}

// ------------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

bool make_map_2d(CUtensorMap* m, void* base, uint64_t inner, uint64_t outer, uint64_t row_bytes, uint32_t box_inner,
                 uint32_t box_outer, CUtensorMapSwizzle sw) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BT>
fd_status launch_tc(fd_ctx* c, const CUtensorMap& mr, const CUtensorMap& mc, const TcParams& p, int grid) {
    const int smem = Smem::total(p.K16);
    if (smem > 227 * 1024) return fail(c, FD_ERR_UNSUPPORTED, "tensor-core kernel needs %d B of shared memory", smem);
    // the attribute is per device: set it on every launch (cheap) rather than remembering one device
    FD_CUDA(c, cudaFuncSetAttribute(k_tc<BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    k_tc<BT><<<grid, kThreads, smem, c->stream>>>(mr, mc, p);
    FD_LAUNCH_CHECK(c, "k_tc");
    return FD_OK;
}

}  // namespace

bool tc_supported(const fd_ctx* c, const ApplyArgs& a) {
    const Layout& L = c->L;
    if (!c->centered) return false;
    if (L.K16 > 4) return false;                                   // D <= 60
    if ((int64_t)L.K16 * L.NP >= ((int64_t)1 << 31)) return false;    // TMA row coordinates are 32-bit
    if (a.Nrow > L.N) return false;
    // The decision depends only on the data set, the bandwidth and the precision mode -- never on the kind of pass --
    // so the degree passes and the block products of one operator always run on the same kernel family (their
    // common rounding bias then cancels in diag(s) K diag(s)).
    // small problems: the split direct-difference kernel fills the GPU better (it covers D <= 32 only)
    if (c->opt_path != FD_PATH_TC && L.N < 16384 && L.DP <= 32) return false;
    const double bprime = a.beta * kLog2e;
    // exponent magnitude the fp16 hi/lo norm pieces and the fp32 Gram accumulation can carry accurately
    const double mag = bprime * (a.rows_are_ctx ? c->max_sq : std::max(c->max_sq, c->row_max_sq));
    if (!(mag < (a.prec == FD_PREC_FAST ? 2000.0 : c->opt_tc_max_mag))) return false;
    if (a.V == nullptr && a.right != nullptr && (!a.right_pos || a.rowsq)) return false;   // (row sums with squares carry no weights)
    return true;
}

fd_status apply_tc(fd_ctx* c, const ApplyArgs& a) {
    const Layout& L = c->L;
    const int64_t N = L.N, NP = L.NP;
    if (!encode_fn()) return fail(c, FD_ERR_CUDA, "cuTensorMapEncodeTiled entry point unavailable");
    FD_TRY(note_capture(c));
    const double bprime = a.beta * kLog2e;
    const bool rowsum = a.V == nullptr;
    const double* mu = c->at<double>(L.mu);
    __half* xp_col = c->at<__half>(L.xp_col);
    __half* xp_row = c->at<__half>(L.xp_row);
    unsigned int* status = c->at<unsigned int>(L.status);
    const int K16 = L.K16;
    // Symmetric row sums (K = K^T): a square pass over the context's own points whose left and right weights are the same
    // vector (the degree passes) evaluates only the tiles on or above the diagonal.
    const bool sym = rowsum && a.sym_ok && c->opt_sym != 0 && a.rows_are_ctx && a.xrow == c->xs() && a.Nrow == N &&
                     a.left == a.right && L.symsum != 0;
    // operands: columns (role 1) always from the context's points, rows (role 0) from a.xrow.  They are the same for every kind of
    // pass: the S tiles of the degree passes and of the block product are bit-identical, so any rounding bias of the Gram
    // accumulation is common to q, d and K and cancels in diag(s) K diag(s).  The operands of the context's own points stay
    // packed for the bandwidth: the products of a solve reuse them.
    // passes over the context's whole point set may leave out tiles that hold no near pair (fd_order.cu)
    const bool all_rows = a.rows_are_ctx && a.xrow == c->xs() && a.Nrow == N;
    const bool prunes = all_rows && !c->sh.on && (rowsum ? sym : a.prec == FD_PREC_FP32);
    // The decision reads a count back.  Degree passes return host scalars and wait anyway, so they decide for the products at their
    // bandwidth too (once: the lists themselves are remade by the first product); any other pass returns without waiting and, at
    // a bandwidth that is not decided, runs over all tiles.
    if (prunes && a.decide && a.prec == FD_PREC_FP32 && c->lists[0].beta != a.beta) FD_TRY(tile_lists(c, a.beta, 0, true));
    if (prunes) FD_TRY(tile_lists(c, a.beta, !rowsum ? 0 : a.rowsq ? 1 : 3, a.decide));
    const bool use_lists = prunes && c->lists[rowsum ? 1 : 0].on && c->lists[rowsum ? 1 : 0].beta == a.beta;
    // The points' order is used, by every Gram-form pass, at the bandwidths that have lists (external rows against ordered columns: neighbouring
    // kernel values alike draw less power; N = 65536, 40009 rows of R^30, 33 vectors: 1.19 ms against 1.23).  At any other bandwidth a pass
    // gives the bits of a context that never made an order.
    const bool ordered = !c->sh.on && ((c->lists[0].on && c->lists[0].beta == a.beta) || (c->lists[1].on && c->lists[1].beta == a.beta));
    const int* col_perm = ordered ? c->at<int>(L.perm) : nullptr;
    const int* row_perm = all_rows ? col_perm : nullptr;
    const PackRole rows{a.xrow, xp_row, a.Nrow, row_perm}, cols{c->xs(), xp_col, N, col_perm};
    const int64_t row0 = a.rows_are_ctx ? (a.xrow - c->xs()) / L.DP : -1;
    const bool have_rows = !c->captured && a.rows_are_ctx && c->packed_row_beta == a.beta && c->packed_row0 == row0 && c->packed_rows == a.Nrow &&
                           c->packed_row_ordered == ordered;
    const bool have_cols = !c->captured && c->packed_beta == a.beta && c->packed_ordered == ordered;
    if (!have_rows || !have_cols) {
        const int first = have_rows ? 1 : 0, roles = (have_rows ? 0 : 1) + (have_cols ? 0 : 1);
        k_pack_points<<<dim3((unsigned)ceil_div(NP, 256), (unsigned)K16, (unsigned)roles), 256, 0, c->stream>>>(
            rows, cols, first, L.DP, c->coords.kept, NP, mu, bprime, std::sqrt(2.0 * bprime), c->coords.kept <= 12 * K16);
        FD_LAUNCH_CHECK(c, "k_pack_points");
        if (!have_rows) {
            c->packed_row_beta = a.rows_are_ctx ? a.beta : -1.0;
            c->packed_row0 = row0; c->packed_rows = a.Nrow; c->packed_row_ordered = ordered;
        }
        c->packed_beta = a.beta; c->packed_ordered = ordered;
    }

    CUtensorMap mr, mc, mh;
    if (!make_map_2d(&mr, xp_row, 32, (uint64_t)K16 * NP, 64, 32, 128, CU_TENSOR_MAP_SWIZZLE_64B) ||
        !make_map_2d(&mc, xp_col, 32, (uint64_t)K16 * NP, 64, 32, 128, CU_TENSOR_MAP_SWIZZLE_64B))
        return fail(c, FD_ERR_CUDA, "cuTensorMapEncodeTiled failed for the point operands");

    TcParams p{};
    p.Nrow = a.Nrow; p.N = N;
    p.num_work = (int)ceil_div(a.Nrow, 256);
    p.num_jt = (int)ceil_div(N, 128);
    // column chunk: ~1024 tiles (40 MB of fp16 operands at b = 64) stay resident in the 126 MB L2 while every CTA sweeps them
    p.jt_chunk = rowsum ? p.num_jt : (c->opt_jt_chunk > 0 ? c->opt_jt_chunk : 1024);
    if (p.jt_chunk > p.num_jt) p.jt_chunk = p.num_jt;
    p.num_chunks = (int)ceil_div(p.num_jt, p.jt_chunk);
    p.np_rows = NP; p.np_cols = NP; p.K16 = K16;
    p.left = a.left; p.status = status; p.perm = row_perm; p.ordered = ordered ? 1 : 0; p.use_lists = use_lists ? 1 : 0;
    const int grid = std::min(p.num_work, c->sm_count);

    if (rowsum && !a.rowsq) {
        float* w = c->at<float>(L.weights);
        k_pad_weights<<<(unsigned)ceil_div(NP, 256), 256, 0, c->stream>>>(a.right, N, NP, col_perm, w);
        FD_LAUNCH_CHECK(c, "k_pad_weights");
        p.weights = w;
    }
    if (rowsum && sym) {
        // the pass with squares notes which tiles hold values that count, for the lists of the pass and the products after it
        const bool note_near = L.near != 0 && ordered && a.rowsq && a.decide && !c->captured && (c->near_beta != a.beta || c->near_direct);
        if (note_near) c->near_beta = -1.0;
        FD_TRY(launch_sym_rowsum(c, mr, mc, p.weights, a.left, a.Y, a.rowsq, row_perm, use_lists, note_near));
        if (note_near) { c->near_beta = a.beta; c->near_direct = false; c->near_unproven = true; }
    } else if (rowsum) {
        p.q = a.Y; p.rowsq = a.rowsq; p.b = 1;
        if (p.rowsq) FD_TRY((launch_tc<16>(c, mr, mc, p, grid)));
        else FD_TRY((launch_tc<32>(c, mr, mc, p, grid)));
    } else {
        __half* wt_hi = c->at<__half>(L.wt_hi);
        float* inv = c->at<float>(L.colscale);
        float* part = c->at<float>(L.part);
        const bool fast = a.prec == FD_PREC_FAST;
        const int vcols = a.ones_last ? a.b - 1 : a.b;
        // column chunks of at most 64, of about equal width (multiples of 16)
        const int cw = fast ? 64 : (int)round_up(ceil_div(a.b, ceil_div(a.b, 64)), 16);
        for (int c0 = 0; c0 < a.b; c0 += cw) {
            const int bc = std::min(cw, a.b - c0);
            const int BT = bc <= 16 ? 16 : bc <= 32 ? 32 : bc <= 48 && !fast ? 48 : 64;
            if (BT > L.BP) return fail(c, FD_ERR_WORKSPACE, "column tile %d wider than the provisioned block buffers (%d)", BT, L.BP);
            const int cm_blocks = (int)std::min<int64_t>(256, ceil_div(N, 1024));
            FD_CUDA(c, launch_behind(c->stream, dim3(cm_blocks, bc), dim3(256), 0, k_colmax_partial, a.V, a.ldv, vcols, a.right, N, c0, part));
            FD_LAUNCH_CHECK(c, "k_colmax_partial");
            FD_CUDA(c, launch_behind(c->stream, dim3((unsigned)std::min<int64_t>(1024, ceil_div(NP, 512)), BT), dim3(256), 0, k_pack_wt,
                                     a.V, a.ldv, vcols, a.right, N, NP, c0, bc, (const float*)part, cm_blocks, inv, wt_hi, fast ? 0 : 1, col_perm));
            FD_LAUNCH_CHECK(c, "k_pack_wt");
            // one map over W_hi (rows 0 .. BT) and, in the fp32-grade mode, W_lo behind it (rows BT .. 2 BT of the same array)
            if (!make_map_2d(&mh, wt_hi, (uint64_t)NP, (uint64_t)(fast ? BT : 2 * BT), (uint64_t)NP * 2, 64, fast ? BT : 2 * BT, CU_TENSOR_MAP_SWIZZLE_128B))
                return fail(c, FD_ERR_CUDA, "cuTensorMapEncodeTiled failed for the block operands");
            p.b = bc; p.colscale_inv = inv; p.Y = a.Y + (int64_t)c0 * a.ldy; p.ldy = a.ldy;
            if (fast) {
                // reduced-precision mode (single fp16 operands): the one-row-tile kernel with sixteen exponential warps
                TcParams pb = p;                   // 128-row work items
                pb.num_work = (int)ceil_div(a.Nrow, 128);
                // the accumulator is flushed every 8 column tiles here: the round-toward-zero loss of the longer groups
                // (a few 1e-6) is far below this mode's own error (3e-4), and the flushes cost 4 %
                pb.flush = c->opt_flush > 0 ? c->opt_flush : 8;
                FD_TRY(launch_fast_product(c, BT, mr, mc, mh, pb, std::min(pb.num_work, c->sm_count)));
                continue;
            }
            p.flush = c->opt_flush > 0 ? c->opt_flush : 1;
            FD_TRY(launch_block_product(c, BT, mr, mc, mh, p));
        }
    }
    return FD_OK;
}

fd_status tc_wait_selftest(fd_ctx* c, long long limit_cycles) {
    k_wait_selftest<<<1, 32, 0, c->stream>>>(c->at<unsigned int>(c->L.status), limit_cycles);
    FD_LAUNCH_CHECK(c, "k_wait_selftest");
    return FD_OK;
}

// Reads the kernel's status word (after the stream has been synchronised by the caller).
fd_status tc_check_status(fd_ctx* c) {
    unsigned int h = 0;
    FD_CUDA(c, cudaMemcpyAsync(&h, c->at<unsigned int>(c->L.status), 4, cudaMemcpyDeviceToHost, c->stream));
    FD_CUDA(c, cudaStreamSynchronize(c->stream));
    if (h != 0) {
        FD_CUDA(c, cudaMemsetAsync(c->at<unsigned int>(c->L.status), 0, 4, c->stream));
        return fail(c, FD_ERR_TIMEOUT, "tensor-core kernel: bounded wait expired (code 0x%x)", h);
    }
    return FD_OK;
}

}  // namespace fd
