// Internal declarations shared by the translation units of libfd.so.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>
#include <string>

#include "fd.h"

namespace fd {

constexpr double kLog2e = 1.4426950408889634074;

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
inline int64_t ceil_div(int64_t x, int64_t m) { return (x + m - 1) / m; }

// ---- tensor-core path geometry ------------------------------------------------------------
constexpr int kTileM = 128;          // rows per row tile (TMEM lanes)
constexpr int kTileJ = 128;          // columns (points j) per column tile
constexpr int kRowTilesPerCta = 2;   // two row tiles share each staged column tile

// Byte offsets of everything the library keeps inside the caller's workspace.
struct Layout {
    int64_t N = 0; int32_t D = 0, DP = 0, b_max = 0, BP = 0, m_max = 0;
    int64_t NP = 0;                  // N rounded up to the tensor-core column tile
    int32_t K16 = 0;                 // 16-wide K slabs of the augmented Gram operand
    size_t xs = 0, xrow = 0, mu = 0, q = 0, d = 0, s = 0, w = 0, rowsq = 0, sums = 0;
    size_t wp = 0;                   // N x BP block of scratch (numerators and denominator of the out-of-sample extension)
    size_t part = 0, part_floats = 0;
    size_t xp_col = 0, xp_row = 0, wt_hi = 0, wt_lo = 0, colscale = 0, status = 0;
    // order of the points and tile lists of the Gram-form kernels (fd_order.cu); 0: not provisioned for this N (near: for this workspace; all
    // lists then share one buffer)
    size_t perm = 0, boxes = 0, zproj = 0, lists[3] = {0, 0, 0}, list_counts[3] = {0, 0, 0}, near = 0, xord = 0;
    bool direct_lists = false;       // provisioned for the direct-difference kernels as well
    size_t weights = 0;              // NP right weights of a Gram-form row sum
    size_t symsum = 0;               // N 64-bit fixed-point sums of the symmetric row-sum mode
    size_t eig_q = 0, eig_w = 0, eig_x = 0, eig_r = 0, eig_small = 0, eig_small_doubles = 0;
    size_t total = 0;
};
// notes: with the degree passes' notes, a list buffer for every kind of pass and lists of the direct-difference kernels; else one buffer for
// lists by the boxes (Gram form only).
Layout make_layout(int64_t N, int32_t D, int32_t b_max, int32_t m_max, bool notes = true);

// Coordinates the kernels work on (keep[0 .. kept)) and those left out because all points share them, with the shared values.
struct Coords {
    int kept, dropped;
    uint8_t keep[64], drop[64];
    float value[64];
};

}  // namespace fd

struct fd_ctx {
    fd::Layout L;
    char* ws = nullptr;
    cudaStream_t stream = nullptr;
    int device = 0;
    int sm_count = 148;
    int centered = 0;
    double mean_sq = 0.0;            // N^-1 sum |x_i - mu|^2 (Eq. 7)
    double max_sq = 0.0;             // max_i |x_i - mu|^2
    fd::Coords coords{};             // L.DP and L.K16 count the kept coordinates (L.D: the caller's)
    bool row_extra = false;          // the external rows staged most recently differ from the points in a dropped coordinate
    double row_max_sq = 0.0;         // the same maximum over the external rows staged most recently (rectangular products)
    // current operator state (set by fd_degree)
    bool have_s = false;
    double beta = 0.0, alpha = 0.0;
    // what the tensor-core operands hold: bandwidth of the unweighted column operand, of the unweighted row operand and its rows
    // (-1: something else)
    double packed_beta = -1.0, packed_row_beta = -1.0;
    int64_t packed_row0 = 0, packed_rows = 0;
    bool packed_ordered = false, packed_row_ordered = false;     // they hold the points in the order of L.perm
    int order_state = 0;             // 1: L.perm holds an order of the points; -1: none will be made
    // tile lists, for Gram-form block products (0) and degree passes (1) and all passes of the direct-difference kernels (2): bandwidth they were decided for, whether
    // they leave out enough to be used, entries in all (products: of the list they go by)
    struct { double beta = -1.0; bool on = false; int64_t total = 0; } lists[3];
    // A pass of this context was recorded into a CUDA graph (set by note_capture, for good).  What the workspace holds is then known to nobody
    // on the host: recording runs nothing, and a replay packs and lists again.  Every pass packs and lists for itself from then on.
    bool captured = false;
    unsigned int direct_epoch = 0;   // number of the latest listed pass of the direct-difference kernels
    double refused_beta = 0.0;       // largest bandwidth at which an order was tried and left out too little
    struct { int kind = -1; double beta = -1.0; } listed[3];     // what the list buffers hold: of the products (0), of the first (1) and the second degree pass (2; Gram form)
    int boxes_kind = -1;
    // bandwidth whose near tiles a degree pass noted in L.near (fd_order.cu).  No pass writes notes once products have been recorded: a
    // replay lists by what they say.
    double near_beta = -1.0;
    bool near_direct = false;        // (by a direct-difference pass)
    bool near_unproven = false;      // the pass that took them has not been seen to finish: a pass that gives up leaves tiles unnoted
    // options
    int opt_path = FD_PATH_AUTO;
    int opt_splits = 0;
    int opt_flush = 0;
    int opt_tail_split = 1;          // (accepted, without effect)
    int opt_sym = 1;                 // symmetric half-work degree passes on the Gram-form kernels (0 = evaluate every tile)
    int opt_jt_chunk = 0;            // column tiles per L2-resident chunk of the tensor-core block product (0 = default)
    int last_path = 0;               // kernel family that served the most recent quadratic pass (FD_PATH_SIMT / FD_PATH_TC)
    fd_precision eigs_prec = FD_PREC_FP32;   // precision mode of fd_eigs's block products (set per stage by the cascade)
    double opt_tc_max_mag = 72.0;    // largest beta' * max|x - mu|^2 the Gram-form kernel is trusted with in fp32 mode
    std::string err;
    // page-locked host memory of the eigensolver: a ring of slots for its small uploads, then the projections, which kernels write
    // there directly (one allocation, made by the first fd_eigs and freed by fd_destroy)
    static constexpr int kStageSlots = 4;
    float* stage = nullptr;
    double* h_out = nullptr;
    cudaEvent_t stage_ev[kStageSlots] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t apply_ev[2] = {nullptr, nullptr};        // around the latest products of a solve
    size_t stage_floats = 0;         // per slot
    size_t h_out_doubles = 0;
    // row-sharded operation (fd_set_shard): this rank owns rows [r0, r1) of every quadratic pass
    struct Shard {
        bool on = false;
        fd_shard h{};                // callbacks, rank, world, exchange buffer
        int64_t chunk = 0, r0 = 0, r1 = 0;
    } sh;
    int64_t row0() const { return sh.on ? sh.r0 : 0; }
    int64_t rows() const { return sh.on ? sh.r1 - sh.r0 : L.N; }

    template <class T> T* at(size_t off) const { return reinterpret_cast<T*>(ws + off); }
    float* xs() const { return at<float>(L.xs); }
    float* q() const { return at<float>(L.q); }
    float* d() const { return at<float>(L.d); }
    float* s() const { return at<float>(L.s); }
    float* w() const { return at<float>(L.w); }
};

namespace fd {

extern int64_t g_launches;           // kernels launched by this library in this process

fd_status fail(fd_ctx* c, fd_status st, const char* fmt, ...);
fd_status cuda_fail(fd_ctx* c, cudaError_t e, const char* what);
#define FD_CUDA(ctx, call)                                                     \
    do {                                                                       \
        cudaError_t e__ = (call);                                              \
        if (e__ != cudaSuccess) return fd::cuda_fail((ctx), e__, #call);       \
    } while (0)
#define FD_TRY(expr)                                                           \
    do {                                                                       \
        fd_status st__ = (expr);                                               \
        if (st__ != FD_OK) return st__;                                        \
    } while (0)
#define FD_LAUNCH_CHECK(ctx, name)                                             \
    do {                                                                       \
        ++fd::g_launches;                                                      \
        cudaError_t e__ = cudaGetLastError();                                  \
        if (e__ != cudaSuccess) return fd::cuda_fail((ctx), e__, name);        \
    } while (0)

// ---- setup (fd_setup.cu) --------------------------------------------------------------------
// Copies X (row-major, pitch ldx) into the padded N x DP layout, computes column means in fp64,
// and mean / max of |x - mu|^2.  Synchronises.
fd_status setup_points(fd_ctx* c, const float* X_dev, int64_t ldx);
// Padded copy of an external row set into the row scratch (rows [r0, r0 + n)).
fd_status stage_rows(fd_ctx* c, const float* Xrow_dev, int64_t ldxrow, int64_t r0, int64_t n);

// Left scaling of a rectangular product over the rows staged most recently: left_i exp(-beta e_i), e_i = the row's squared distance
// from the points in the dropped coordinates; *out = left itself when all e_i are 0.
fd_status row_factor(fd_ctx* c, const float* left, double beta, int64_t n, const float** out);

// ---- quadratic passes -----------------------------------------------------------------------
// General product on rows [0, Nrow) of `xrow` (padded N x DP layout, device) against the context's
// points:  Y = diag(left) K diag(right) V.  V == nullptr means the ones vector (b = 1).
struct ApplyArgs {
    const float* xrow; int64_t Nrow;        // padded row points (SIMT layout, uncentred)
    bool rows_are_ctx;                      // xrow is the context's own point set
    double beta;
    const float* left; const float* right;  // may be null
    const float* V; int64_t ldv; int32_t b;
    float* Y; int64_t ldy;
    double* rowsq;                          // optional: sum_j K_ij^2 per row (rowsum mode, b = 1, V null)
    bool ones_last;                         // block mode: column b - 1 of the block is the ones vector, V holds the others
    bool right_pos;                         // caller guarantees right > 0 elementwise
    bool sym_ok;                            // square pass with left == right, weights in (0, 1]: the symmetric half-work row sums may serve it
    bool decide;                            // the pass may wait for the decision which tiles a bandwidth leaves out (degree passes: they wait anyway)
    fd_precision prec;
};
fd_status apply_simt(fd_ctx* c, const ApplyArgs& a);
fd_status apply_tc(fd_ctx* c, const ApplyArgs& a);
bool tc_supported(const fd_ctx* c, const ApplyArgs& a);
fd_status apply_dispatch(fd_ctx* c, const ApplyArgs& a);
// Argument checks of a block, and of a product's two blocks of b columns (which must not overlap).
fd_status check_block(fd_ctx* c, const float* p, int64_t ld, int64_t rows, const char* what);
fd_status check_in_out(fd_ctx* c, const float* V, int64_t ldv, int64_t vrows, const float* Y, int64_t ldy, int64_t yrows, int32_t b);
// Body of fd_apply_general with one more promise: right_pos = the caller guarantees right > 0 elementwise, which lets a
// row-sum (V == nullptr) with a right vector take the same kernel family as the block products of the same operator.
fd_status apply_general(fd_ctx* c, double beta, const float* left_dev, const float* right_dev, bool right_pos,
                        const float* Xrow_dev, int64_t Nrow, int64_t ldxrow, const float* V_dev, int64_t ldv, int32_t b,
                        float* Y_dev, int64_t ldy, fd_precision prec, bool gather_out = true);

// ---- row-sharded operation (fd_shard.cu) ----------------------------------------------------------
// Rows [begin, end) of rank `rank`: contiguous ranges of round_up(ceil(N / world), 256) rows.
void shard_range(int64_t N, int world, int rank, int64_t* begin, int64_t* end);
// A is column-major with pitch lda and `cols` columns; on entry every rank holds valid values in its own rows, on
// return in all N rows.  No-op for an unsharded context.  cols is split into groups of at most b_max internally.
fd_status gather_rows(fd_ctx* c, float* A, int64_t lda, int cols);
// In-place sum over the ranks of n host doubles.  No-op for an unsharded context.
fd_status allreduce_host(fd_ctx* c, double* buf, int64_t n);
// Sets c->captured if the context's stream is being captured: for passes that would rely on what an earlier one left in the workspace.
fd_status note_capture(fd_ctx* c);
// Tile lists of a bandwidth for c->lists[kind] (fd_order.cu): decides c->lists[kind] and, where they are
// used, brings them into the workspace; orders the points first if that can pay.  A new bandwidth is decided, with a wait, only where
// `decide` allows it; without, nothing is listed for it.
fd_status tile_lists(fd_ctx* c, double beta, int kind, bool decide);
// Reads and clears the tensor-core kernel's status word; FD_ERR_TIMEOUT if a bounded wait expired.  Synchronises.
fd_status tc_check_status(fd_ctx* c);
// Launches a one-thread kernel whose bounded wait must expire after limit_cycles (test of the time-out plumbing).
fd_status tc_wait_selftest(fd_ctx* c, long long limit_cycles);

// ---- small kernels (fd_elementwise.cu) ------------------------------------------------------
fd_status ew_pow(fd_ctx* c, const float* in, double p, float* out, int64_t n);            // out = in^p
// s = qa * d^-1/2 (qa null: 1); also copies q, d, s to the outputs that are not null.
fd_status ew_scale_vec(fd_ctx* c, const float* qa, const float* q, const float* d, float* s, int64_t n, float* q_out, float* d_out, float* s_out);
// Deterministic fp64 sums of a float vector and a double vector (two-stage tree) -> out_dev[0], out_dev[1].
fd_status reduce_sums(fd_ctx* c, const float* q, const double* rowsq, int64_t n, double* out_dev);
fd_status scale_cols_by_pow(fd_ctx* c, const float* v, int64_t ldv, int32_t cols, const float* d, double p,
                            float* out, int64_t ldout, int64_t n);

}  // namespace fd

#ifdef __CUDACC__
#include <utility>

namespace fd {

// Launches a kernel that may start while the kernel before it in the stream ends: it calls grid_wait() in every thread before it touches memory
// (also in blocks that have nothing to do: what follows waits for this kernel only).  grid_go() lets the one after it do the same.
template <class... Params, class... Args>
cudaError_t launch_behind(cudaStream_t stream, dim3 grid, dim3 block, size_t smem, void (*kernel)(Params...), Args&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream; cfg.attrs = &attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
__device__ __forceinline__ void grid_wait() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void grid_go() { cudaTriggerProgrammaticLaunchCompletion(); }

// Two fp32 values in a register pair: an instruction on both takes one issue slot and the time of two on the FMA pipe.
__device__ __forceinline__ uint64_t pair2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 split2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

}  // namespace fd
#endif
