// fd_eigs: leading eigenpairs of M = diag(s) K diag(s) (Eq. 2) by block Krylov / Rayleigh-Ritz
// with residual expansion and thick restart.
//
// The paper names "block implicitly restarted Lanczos" (Sec. 2.3) and gives no detail, so the
// scheme is fixed here.  An orthonormal basis Q (N x m) is kept together with its image
// W = M Q and the projections T = Q^T W, G = Q^T Q (fp64).  A Rayleigh-Ritz step gives Ritz pairs, explicit residuals
// R_i = W x_i - theta_i Q x_i for the leading k + 1 + buffer pairs, and the b residuals of largest
// norm as the next block.  A block is orthogonalised against Q and within itself (eigen-based, drops dependent directions),
// appended, and M is applied to it only.  The blocks after it continue the Krylov space of the newest one (M times the last
// block, block Lanczos with full orthogonalisation) until the next Rayleigh-Ritz step: in exact arithmetic the residuals of all
// Ritz vectors lie in the span of that continuation, so the space grows the same way (measured: the same number of products
// within one or two), while the projected eigenproblem (host) and the residual passes (O(N m k)) are paid once in about four products.
// For a cold one-block start this spans the block Krylov space of block Lanczos; unlike the three-term
// recurrence it accepts an arbitrary warm-start basis.
// When the basis is full it is compressed onto the leading Ritz vectors (thick restart).
// The Perron vector sqrt(d) / |sqrt(d)| is known in closed form and always seeds the basis.
// Vectors are fp32; every inner product and the small eigenproblem are fp64, and the measured
// Gram matrix Q^T Q corrects the projected problem to first order, so fp32 loss of
// orthogonality does not reach the Ritz values.
//
// What bounds it: the products with M at N >= 2^17; below, the host waits of a step (two: the projections of the new block
// and of its first orthogonalisation) and the launches between them.  A step costs two A^T B passes, two A S passes and one product.
// N = 16384 (R^4, k = 32, b = 16): 87 -> 45 ms; N = 65536 (R^30, k = 32, b = 32): 64 -> 45 ms; N = 2^17 (R^12, k = 64, b = 32): 457 -> 355 ms
// against a Rayleigh-Ritz step per product with separate passes for every projection.
//
// Row-sharded contexts: every rank keeps rows [r0, r0 + n) of Q, W and the work blocks (pitch N, same addresses as
// the unsharded layout), all tall-skinny products run on those rows, every reduced quantity
// is summed over the ranks on the host (so all ranks take the same decisions), and the rows of a new block are gathered
// from their owners before M is applied to it.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "fd_dense.h"

namespace fd {

namespace {

using clk = std::chrono::steady_clock;
inline double secs(clk::time_point a, clk::time_point b) { return std::chrono::duration<double>(b - a).count(); }

struct Solver {
    fd_ctx* c;
    int64_t N;                      // pitch of every tall matrix = number of points
    int64_t r0, n;                  // rows this rank owns (0, N unless the context is row-sharded)
    int m_cap, BP;
    float *Q, *W, *X;               // N x m_cap each (X = spare for out-of-place updates and the residuals)
    float* R;                       // N x BP
    float* d_S;                     // device: small right factors
    double* d_scr; size_t scr_n;    // device: partials of the projections
    size_t S_floats;                // capacity of d_S and of a staging slot
    std::vector<double> T, G;       // host, column-major, pitch m_cap
    double* h = nullptr;            // page-locked result of the latest projection
    volatile unsigned int* h_status = nullptr;   // page-locked copy of the tensor-core kernels' status word
    int stage_next = 0;             // next slot of the context's staging ring
    int m = 0;
    int applies = 0, restarts = 0;
    double t_apply = 0.0;
    bool clean = true;              // the latest block was far from dependent: one orthogonalisation was enough
    bool timing = false;            // the events around the latest products are not read yet

    Panel own(const float* p, int cols) const { return panel(p + r0, cols, N); }
    Panel own(const float* p1, int c1, const float* p2, int c2) const { return panel(p1 + r0, c1, p2 + r0, c2, N); }

    // The page-locked buffers live in the context (allocated once): an upload never waits for the stream unless its slot is
    // still in flight.
    fd_status init_staging(size_t out_doubles) {
        if (c->stage_floats < S_floats || c->h_out_doubles < out_doubles) {
            FD_CUDA(c, cudaStreamSynchronize(c->stream));
            if (c->stage) { FD_CUDA(c, cudaFreeHost(c->stage)); c->stage = nullptr; c->stage_floats = 0; c->h_out_doubles = 0; }
            const size_t slot = (size_t)round_up((int64_t)S_floats, 64);
            FD_CUDA(c, cudaMallocHost(reinterpret_cast<void**>(&c->stage), sizeof(float) * slot * fd_ctx::kStageSlots + sizeof(double) * (out_doubles + 1)));
            c->stage_floats = slot;
            c->h_out = reinterpret_cast<double*>(c->stage + slot * fd_ctx::kStageSlots);
            c->h_out_doubles = out_doubles;
            for (int i = 0; i < fd_ctx::kStageSlots; ++i)
                if (!c->stage_ev[i]) FD_CUDA(c, cudaEventCreateWithFlags(&c->stage_ev[i], cudaEventDisableTiming));
            for (int i = 0; i < 2; ++i)
                if (!c->apply_ev[i]) FD_CUDA(c, cudaEventCreate(&c->apply_ev[i]));
        }
        h = c->h_out;
        h_status = reinterpret_cast<unsigned int*>(c->h_out + c->h_out_doubles);
        *h_status = 0;
        return FD_OK;
    }
    // Slot for a right factor of `floats` entries: the caller fills it and sends it.
    fd_status stage_slot(size_t floats, float** p) {
        if (floats > S_floats) return fail(c, FD_ERR_WORKSPACE, "staging buffer too small for a right factor");
        FD_CUDA(c, cudaEventSynchronize(c->stage_ev[stage_next]));     // the copy that used this slot last (four uploads ago) has finished
        *p = c->stage + c->stage_floats * stage_next;
        return FD_OK;
    }
    fd_status send_slot(size_t floats) {
        FD_CUDA(c, cudaMemcpyAsync(d_S, c->stage + c->stage_floats * stage_next, sizeof(float) * floats, cudaMemcpyHostToDevice, c->stream));
        FD_CUDA(c, cudaEventRecord(c->stage_ev[stage_next], c->stream));
        stage_next = (stage_next + 1) % fd_ctx::kStageSlots;
        return FD_OK;
    }
    // Waits for the projection written to h (cnt doubles) and sums it over the ranks.
    fd_status fetch(int64_t cnt) {
        FD_CUDA(c, cudaStreamSynchronize(c->stream));
        if (timing) {
            float ms = 0.f;
            FD_CUDA(c, cudaEventElapsedTime(&ms, c->apply_ev[0], c->apply_ev[1]));
            t_apply += 1e-3 * ms;
            timing = false;
        }
        FD_TRY(allreduce_host(c, h, cnt));
        // the status word of the products before this wait (the sum above first: every rank takes that step)
        if (*h_status != 0) return tc_check_status(c);
        return FD_OK;
    }
    // h = A^T B (column-major, pitch = columns of A)
    fd_status project(const Panel& A, const Panel& B) {
        const int64_t cnt = (int64_t)(A.m1 + A.m2) * (B.m1 + B.m2);
        if ((size_t)cnt > c->h_out_doubles) return fail(c, FD_ERR_WORKSPACE, "projection larger than its buffer");
        FD_TRY(tn_product(c, A, B, n, h, d_scr, scr_n));
        return fetch(cnt);
    }

    // W[:, c0 : c0 + n) = M Q[:, c0 : c0 + n).
    fd_status apply_cols(int c0, int cnt, int bw) { return apply_block(Q + (int64_t)c0 * N, W + (int64_t)c0 * N, cnt, bw); }
    // out = M B for cnt columns, in blocks of at most bw.  Nothing waits for the products here: their time is read
    // after the wait of the projection that follows.
    fd_status apply_block(float* B, float* out, int cnt, int bw) {
        FD_CUDA(c, cudaEventRecord(c->apply_ev[0], c->stream));
        FD_TRY(gather_rows(c, B, N, cnt));                           // the product needs all rows of the right block
        for (int o = 0; o < cnt; o += bw) {
            int w = std::min(bw, cnt - o);
            FD_TRY(apply_general(c, c->beta, c->s(), c->s(), false, nullptr, N, 0, B + (int64_t)o * N, N, w,
                                 out + (int64_t)o * N, N, c->eigs_prec, /*gather_out=*/false));
            ++applies;
        }
        // (looked at after the next projection's wait)
        if (c->last_path == FD_PATH_TC)
            FD_CUDA(c, cudaMemcpyAsync(const_cast<unsigned int*>(h_status), c->at<unsigned int>(c->L.status), 4, cudaMemcpyDeviceToHost, c->stream));
        FD_CUDA(c, cudaEventRecord(c->apply_ev[1], c->stream));
        timing = true;
        return FD_OK;
    }

    // Recompute T = Q^T W and G = Q^T Q for the first m columns.
    fd_status full_projection() {
        const int step = std::max(1, (int)std::min<size_t>((size_t)m, scr_n / (size_t)m));
        for (int pass = 0; pass < 2; ++pass) {
            std::vector<double>& D = pass ? G : T;
            for (int j0 = 0; j0 < m; j0 += step) {
                const int w = std::min(step, m - j0);
                FD_TRY(project(own(Q, m), own((pass ? Q : W) + (int64_t)j0 * N, w)));
                for (int j = 0; j < w; ++j)
                    for (int i = 0; i < m; ++i) D[i + (size_t)(j0 + j) * m_cap] = h[i + (size_t)j * m];
            }
            for (int j = 0; j < m; ++j)
                for (int i = 0; i < j; ++i) {
                    const double v = 0.5 * (D[i + (size_t)j * m_cap] + D[j + (size_t)i * m_cap]);
                    D[i + (size_t)j * m_cap] = D[j + (size_t)i * m_cap] = v;
                }
        }
        return FD_OK;
    }

    // After p columns were appended at position m (their images in W): fills the new rows / columns of T and G.  On return
    // h holds [Q W_new]^T [Q_new W_new] with Q including the new columns (m + p rows) -- the projection that the block
    // W_new needs when it becomes the next expansion.
    fd_status extend_projection(int p) {
        const int mt = m + p, rows = mt + p;
        const float *Qn = Q + (int64_t)m * N, *Wn = W + (int64_t)m * N;
        FD_TRY(project(own(Q, mt, Wn, p), own(Qn, p, Wn, p)));
        for (int pass = 0; pass < 2; ++pass) {
            std::vector<double>& D = pass ? G : T;
            const double* z = h + (size_t)(pass ? 0 : p) * rows;
            for (int j = 0; j < p; ++j)
                for (int i = 0; i < mt; ++i) {
                    double v = z[i + (size_t)j * rows];
                    if (i >= m) v = 0.5 * (v + z[(m + j) + (size_t)(i - m) * rows]);
                    D[i + (size_t)(m + j) * m_cap] = v;
                    D[(m + j) + (size_t)i * m_cap] = v;
                }
        }
        m = mt;
        return FD_OK;
    }

    // F (p x rank, column-major) turns the columns whose p x p Gram matrix is g (column-major, overwritten) into orthonormal ones.  By
    // Cholesky if every pivot of the matrix scaled to a unit diagonal exceeds kGoodPivot, else by its eigen-decomposition, leaving
    // out directions with an eigenvalue at or below drop_tol.  lam_min: about the smallest eigenvalue kept.
    static constexpr double kGoodPivot = 0.1;
    fd_status orthonormal_factor(double* g, int p, double drop_tol, std::vector<double>& F, int& rank, double& lam_min) {
        std::vector<double> dinv(p);
        for (int j = 0; j < p; ++j) {
            const double dj = g[j + (size_t)j * p];
            dinv[j] = dj > 1e-60 ? 1.0 / std::sqrt(dj) : 0.0;
        }
        for (int j = 0; j < p; ++j)
            for (int i = 0; i <= j; ++i) {
                const double v = 0.5 * (g[i + (size_t)j * p] + g[j + (size_t)i * p]) * dinv[i] * dinv[j];
                g[i + (size_t)j * p] = g[j + (size_t)i * p] = v;
            }
        // well-conditioned (the usual case): Cholesky g = L L^T, F = D^-1/2 L^-T; its pivots bound how close to dependent the columns are
        {
            std::vector<double> Lc((size_t)p * p, 0.0);
            bool good = true;
            for (int j = 0; j < p && good; ++j) {
                for (int i = j; i < p; ++i) {
                    double v = g[i + (size_t)j * p];
                    for (int l = 0; l < j; ++l) v -= Lc[(size_t)i * p + l] * Lc[(size_t)j * p + l];
                    if (i == j) {
                        good = v > kGoodPivot;
                        if (!good) break;
                        Lc[(size_t)j * p + j] = std::sqrt(v);
                    } else Lc[(size_t)i * p + j] = v / Lc[(size_t)j * p + j];
                }
            }
            if (good) {
                F.assign((size_t)p * p, 0.0);                      // column j of L^-T: back substitution against e_j
                for (int j = 0; j < p; ++j) {
                    double* f = &F[(size_t)j * p];
                    for (int i = j; i >= 0; --i) {
                        double v = i == j ? 1.0 : 0.0;
                        for (int l = i + 1; l <= j; ++l) v -= Lc[(size_t)l * p + i] * f[l];
                        f[i] = v / Lc[(size_t)i * p + i];
                    }
                    for (int i = 0; i <= j; ++i) f[i] *= dinv[i];
                }
                rank = p;
                lam_min = kGoodPivot;
                return FD_OK;
            }
        }
        std::vector<double> lam, U;
        if (!sym_eig(g, p, lam, U)) return fail(c, FD_ERR_NOT_CONVERGED, "small eigenproblem (orthonormalise) failed");
        rank = 0;
        lam_min = 1.0;
        F.clear();
        for (int j = p - 1; j >= 0; --j) {
            if (!(lam[j] > drop_tol)) continue;
            const double f = 1.0 / std::sqrt(lam[j]);
            for (int i = 0; i < p; ++i) F.push_back(dinv[i] * U[i + (size_t)j * p] * f);
            lam_min = lam[j];
            ++rank;
        }
        return FD_OK;
    }

    // Orthonormalise the p columns of B (pitch N) among themselves.  Result in B, p updated.
    fd_status orthonormalise(float*& B, float*& spare, int& p, double drop_tol) {
        if (p == 0) return FD_OK;
        FD_TRY(project(own(B, p), own(B, p)));
        std::vector<double> g(h, h + (size_t)p * p), F;
        int rank; double lam_min;
        FD_TRY(orthonormal_factor(g.data(), p, drop_tol, F, rank, lam_min));
        if (rank == 0) { p = 0; return FD_OK; }
        float* S = nullptr;
        FD_TRY(stage_slot(F.size(), &S));
        for (size_t i = 0; i < F.size(); ++i) S[i] = (float)F[i];
        FD_TRY(send_slot(F.size()));
        FD_TRY(nn_product(c, own(B, p), d_S, p, rank, spare + r0, N, n));
        std::swap(B, spare);
        p = rank;
        return FD_OK;
    }

    // dst = (B - Q C) F for p columns B and the basis Q[:, 0 : m): z = [Q B]^T B holds C (rows 0 .. m, pitch ldz); F is p x pk.
    fd_status subtract_and_mix(const float* B, int p, const double* z, int ldz, const double* F, int pk, float* dst) {
        float* S = nullptr;
        const size_t cnt = (size_t)(m + p) * pk;
        FD_TRY(stage_slot(cnt, &S));
        std::vector<double> col(m);
        for (int j = 0; j < pk; ++j) {
            const double* f = F + (size_t)j * p;
            std::fill(col.begin(), col.end(), 0.0);
            for (int l = 0; l < p; ++l) {
                const double fl = f[l];
                if (fl == 0.0) continue;
                host_axpy(col.data(), z + (size_t)l * ldz, -fl, m);
            }
            for (int i = 0; i < m; ++i) S[i + (size_t)j * (m + p)] = (float)col[i];
            for (int l = 0; l < p; ++l) S[m + l + (size_t)j * (m + p)] = (float)f[l];
        }
        FD_TRY(send_slot(cnt));
        return nn_product(c, own(Q, m, B, p), d_S, m + p, pk, dst + r0, N, n);
    }

    // Orthonormalises the block B (p <= BP columns, not inside Q's first m columns) against the basis and within itself; the
    // result goes to `target` and p is updated (0: nothing new).  other: scratch of the same size (B may be it).
    // z: [Q B]^T B of pitch ldz if the caller has it, else null.
    //   1. R = (B - Q C) scaled to unit columns: removes the basis to fp32 rounding of B's own size;
    //   2. Q_new = (R - Q C') F with C' = Q^T R (small now) and F from R^T R - C'^T C', which is accurate because C' is small;
    //   3. once more if the block was nearly dependent, so that step 2's rounding was magnified.
    fd_status expand(const float* B, int& p, const double* z, int ldz, float* target, float* other) {
        if (p == 0) return FD_OK;
        std::vector<double> F;
        if (!z) {
            FD_TRY(project(own(Q, m, B, p), own(B, p)));
            z = h; ldz = m + p;
        }
        F.assign((size_t)p * p, 0.0);
        for (int j = 0; j < p; ++j) {
            const double* zj = z + (size_t)j * ldz;
            double d = zj[m + j], cc = 0.0;
            for (int i = 0; i < m; ++i) cc += zj[i] * zj[i];
            const double left = std::max(d - cc, 1e-12 * d);      // |column|^2 after the projection (floor: cancellation)
            F[j + (size_t)j * p] = left > 1e-60 ? 1.0 / std::sqrt(left) : 0.0;
        }
        float* dst = B == other ? target : other;
        FD_TRY(subtract_and_mix(B, p, z, ldz, F.data(), p, dst));
        for (int pass = 0; pass < 2; ++pass) {
            const float* src = dst;
            FD_TRY(project(own(Q, m, src, p), own(src, p)));
            const int ld = m + p;
            std::vector<double> g((size_t)p * p);
            double cmax = 0.0;
            for (int j = 0; j < p; ++j)
                for (int i = 0; i < p; ++i) {
                    const double *ci = h + (size_t)i * ld, *cj = h + (size_t)j * ld;
                    double v = cj[m + i];
                    for (int l = 0; l < m; ++l) v -= ci[l] * cj[l];
                    g[i + (size_t)j * p] = v;
                    if (i == 0) for (int l = 0; l < m; ++l) cmax = std::max(cmax, std::fabs(cj[l]) / std::sqrt(std::max(cj[m + j], 1e-60)));
                }
            int rank; double lam_min;
            FD_TRY(orthonormal_factor(g.data(), p, pass == 0 ? 1e-5 : 1e-3, F, rank, lam_min));
            if (rank == 0) { p = 0; return FD_OK; }
            dst = src == other ? target : other;
            FD_TRY(subtract_and_mix(src, p, h, ld, F.data(), rank, dst));
            p = rank;
            clean = pass == 0 && lam_min > 1e-2 && cmax < 1e-2;
            if (clean) break;
        }
        if (dst == other) FD_TRY(copy_cols(c, other + r0, N, target + r0, N, p, n));
        return FD_OK;
    }
    fd_status expand(const float* B, int& p, const double* z, int ldz) { return expand(B, p, z, ldz, Q + (int64_t)m * N, R); }
};

}  // namespace
}  // namespace fd

using namespace fd;

extern "C" fd_status fd_eigs(fd_ctx* c, int32_t k, int32_t b, double tol, int32_t max_applies, const float* Q0_dev,
                             int64_t ldq0, int32_t q0_cols, double* evals_host, float* evecs_dev, int64_t ldv,
                             fd_eigs_info* info) {
    if (!c) return FD_ERR_INVALID;
    auto t_start = clk::now();
    const Layout& L = c->L;
    const int64_t N = L.N;
    if (!c->have_s) return fail(c, FD_ERR_INVALID, "fd_eigs before fd_degree");
    if (k < 0 || (int64_t)k + 1 > N) return fail(c, FD_ERR_INVALID, "k + 1 = %d exceeds N or k < 0", k + 1);
    if (b < 1 || b > L.b_max) return fail(c, FD_ERR_INVALID, "b outside 1..b_max");
    if (!(tol > 0) || max_applies < 1 || !evals_host || !evecs_dev || ldv < N) return fail(c, FD_ERR_INVALID, "bad fd_eigs argument");
    if (Q0_dev && (q0_cols < 1 || ldq0 < N)) return fail(c, FD_ERR_INVALID, "bad warm-start basis");
    const int nwant = k + 1;
    if (L.m_max < 2 * nwant + b && L.m_max < N) return fail(c, FD_ERR_WORKSPACE, "m_max = %d < 2 (k + 1) + b = %d", L.m_max, 2 * nwant + b);

    Solver S;
    S.c = c; S.N = N; S.r0 = c->row0(); S.n = c->rows(); S.BP = L.BP;
    const int64_t r0 = S.r0, n = S.n;
    S.m_cap = (int)std::min<int64_t>(L.m_max, N);
    const int m_cap = S.m_cap;
    S.Q = c->at<float>(L.eig_q); S.W = c->at<float>(L.eig_w); S.X = c->at<float>(L.eig_x);
    S.R = c->at<float>(L.eig_r);
    double* small = c->at<double>(L.eig_small);
    const size_t mm = (size_t)L.m_max * std::max(L.m_max, L.BP);
    S.d_S = reinterpret_cast<float*>(small);
    S.S_floats = 2 * mm;
    S.d_scr = small + mm;
    S.scr_n = L.eig_small_doubles - mm;
    S.T.assign((size_t)m_cap * m_cap, 0.0);
    S.G.assign((size_t)m_cap * m_cap, 0.0);
    auto t_i0 = clk::now();
    FD_TRY(S.init_staging(std::max((size_t)m_cap * m_cap, (size_t)(m_cap + 2 * L.BP) * 2 * L.BP)));
    const double t_init = secs(t_i0, clk::now());

    const int buffer = std::min<int>(std::min(b, 8), (int)std::max<int64_t>(0, N - nwant));
    const int nsel_max = nwant + buffer;

    // ---- start basis: Perron vector, then the warm-start columns or a random block ----------
    FD_TRY(sqrt_vec(c, c->d() + r0, S.Q + r0, n));
    int cols = 1;
    const int room = std::max(0, m_cap - b - 1);                 // leave space for one expansion block
    if (Q0_dev) {
        int take = std::min(q0_cols, std::max(room, std::min(m_cap - 1, nwant)));
        take = std::min(take, m_cap - 1);
        FD_TRY(copy_cols(c, Q0_dev + r0, ldq0, S.Q + N + r0, N, take, n));
        cols += take;
    } else {
        int take = std::min(std::max(b, 1), m_cap - 1);
        if (take > 0) FD_TRY(random_fill(c, S.Q + N + r0, N, take, n, r0, 0x5EEDu));
        cols += take;
    }
    {
        // orthonormalise the start block in place (may exceed BP columns: use the spare basis buffer)
        float* B = S.Q; float* spare = S.X; int p = cols;
        // d_S must hold p x p floats: p <= m_cap
        FD_TRY(S.orthonormalise(B, spare, p, 1e-10));
        FD_TRY(S.orthonormalise(B, spare, p, 1e-10));
        S.Q = B; S.X = spare;
        if (p == 0) return fail(c, FD_ERR_NONFINITE, "start basis has no usable column");
        S.m = p;
    }
    FD_TRY(S.apply_cols(0, S.m, b));
    FD_TRY(S.full_projection());

    std::vector<double> theta, Xr;        // Ritz values (descending) and vectors (m x nsel, pitch m)
    std::vector<double> resid;
    int nsel = 0, nconv = 0, nlock = 0;
    fd_status final_status = FD_ERR_NOT_CONVERGED;
    int stagnation = 0;
    // stagnation of the residuals at the accuracy floor of the fp32 operator (noise-smeared spectra): stop early
    double best_res = 1e300;
    int since_best = 0;
    // blocks appended between two Rayleigh-Ritz steps
    // (A basis smaller than three times the wanted pairs has room for two blocks between restarts and cuts into the wanted pairs'
    // clusters.  There every block is a residual block, largest residual first, and a solve that reaches the accuracy floor of the fp32
    // operator is reported as stalled.  Krylov blocks and wanted pairs first need the same number of products there (6-torus, N = 2^17,
    // k = 64, capacity 192: 49 and 49; 2-torus, beta = 30, capacity 98: 66 and 67) and end at another floor, either side of 1e-6.)
    const bool small_basis = m_cap < 3 * nwant && m_cap < N;
    const int kMaxBlocks = small_basis ? 1 : 4;
    const bool wanted_first = !small_basis;
    // Ritz vectors kept at a restart: three fifths of the basis and the room that no whole block fits in.  Fewer, down to twice the wanted pairs, where that
    // leaves the gap between the last wanted Ritz value and the first one not kept: a block or more beyond the next restart for about as
    // many products (6-torus, N = 2^17, k = 64: 11 -> 8 restarts, 293 -> 282 ms; N = 86893, k = 40: 19 -> 12, 153 -> 133 ms; 2-torus, N = 16384,
    // k = 25: 20 -> 12, 28.5 -> 23.5 ms).  Fewer in a cluster that the wanted pairs belong to closes the gap: 6-torus, N = 20000, k = 3, capacity 28:
    // 29 -> 81 products, N = 16384, k = 32, capacity 163: 27 -> 45 (now 31 and 26).  kGap: 0.15 still cuts clusters (32 products), 0.5 and 0.8 keep
    // more than they need (2-torus, k = 32: 25.6 -> 25.8 ms; R^30: 31.0 -> 32.0 at 0.5).
    constexpr double kGap = 0.3;
    const int most_kept = small_basis ? (m_cap * 3) / 5 : m_cap - (m_cap - (m_cap * 3) / 5) / b * b;
    const auto kept_at = [&](const double* ritz, int m) {          // ascending Ritz values of m columns
        const int most = std::min(m - 1, most_kept);
        if (small_basis || m < nwant) return most;
        const double last = ritz[m - nwant], gap = last - ritz[m - 1 - most];
        for (int fewer = m_cap - (m_cap - 2 * nwant) / b * b; fewer < most; fewer += b)
            if (last - ritz[m - 1 - fewer] >= kGap * gap) return fewer;
        return most;
    };
    double last_worst = 0.0, last_rate = 0.0;
    int last_applies = 0;
    // The block after the last one before a Rayleigh-Ritz step is made, and M applied to it, while the host solves the projected
    // eigenproblem: the residuals of all Ritz vectors lie in its span, so it is the next expansion whatever that step decides.  It
    // waits in R and its image in the extension's scratch: the basis may be full.  Only while the blocks are a Krylov sequence (cold starts,
    // from the first step on), and while the residuals are expected to stay well above the tolerance (kAhead): a solve's last steps take
    // explicit residuals, which also see what the stored images have lost to rounding.
    // What the sequence has lost to rounding it never finds again.  A nearly dependent block is mostly rounding in its weak directions, so
    // it ends the sequence (an explicit residual block nearly always is one: smallest eigenvalue 1e-3 to 3e-5 where Krylov blocks have 0.1), and
    // so does a wanted residual of which a part as large as kLost of the worst one lies outside the block's span: that block is still taken,
    // the next one is of explicit residuals.  Without these two, solves stalled at 1e-4 until max_applies (6-torus, N = 2000, k = 23, capacity
    // 328: 120 products and 1 pair where 49 had given 24) or took up to twice the products.
    // 6-torus, N = 2^17, k = 64, capacity 259: 323 -> 293 ms, N = 86893, k = 40: 185 -> 152; R^30, N = 65536, k = 32: 38 -> 32; 2-torus, N = 16384,
    // k = 32: 29.1 -> 26.3.
    constexpr double kAhead = 100.0, kLost = 0.1;
    bool krylov = !Q0_dev && !small_basis;
    float* const ahead_image = c->at<float>(L.wp);
    int ahead = 0;
    // The stored images drift from M Q: a restart rounds Q S and W S separately, and what they differ by ends up in every residual (0.3e-6 to
    // 0.9e-6 after 20 to 100 restarts).  Where the worst wanted residual has not improved by 10 % over kStall products within twice the
    // tolerance, the next restart applies M to the kept basis again.  6-torus, N = 30000, k = 64, capacity 259: 65 of 65 pairs instead of a
    // stall at 1.05e-6 with 13; capacity 195: 0.74e-6 after 87 products instead of 1.18e-6 after 95.  Solves that do not stall never do it.
    constexpr int kStall = 8, kMaxRefreshes = 2;
    int refreshes = 0;

    double t_rr = 0, t_eig = 0, t_res = 0, t_restart = 0, t_orth = 0, t_ext = 0;
    for (int iter = 0;; ++iter) {
        const int m = S.m;
        auto tp0 = clk::now();
        // ---- Rayleigh-Ritz with first-order correction for G = Q^T Q = I + E ---------------------
        // Tc = T - (E T + T E) / 2 with E = G - I; T E = (E T)^T because both are symmetric
        std::vector<double> Tc((size_t)m * m), ET((size_t)m * m, 0.0);
#pragma omp parallel for schedule(static) if (m >= 64)
        for (int j = 0; j < m; ++j)
            for (int l = 0; l < m; ++l) {
                const double t = S.T[l + (size_t)j * m_cap];
                const double* Ecol = &S.G[(size_t)l * m_cap];
                double* o = &ET[(size_t)j * m];
                host_axpy(o, Ecol, t, m);                                 // G column l ...
                o[l] -= t;                                                 // ... minus the identity
            }
        for (int j = 0; j < m; ++j)
            for (int i = 0; i < m; ++i)
                Tc[i + (size_t)j * m] = S.T[i + (size_t)j * m_cap] - 0.5 * (ET[i + (size_t)j * m] + ET[j + (size_t)i * m]);
        std::vector<double> lam, U;
        auto tp1 = clk::now();
        // eigenvectors: the leading Ritz vectors on every step; the larger kept set only when this step may restart
        const int nvec_ritz = std::min(nsel_max, m);
        const bool may_restart = m + b > m_cap;
        const int nvec = may_restart ? std::max(nvec_ritz, std::min(m - 1, most_kept)) : nvec_ritz;
        const auto needed = [&](const double* l) { return may_restart ? std::max(nvec_ritz, kept_at(l, m)) : nvec; };
        if (!sym_eig(Tc.data(), m, lam, U, nvec, needed)) return fail(c, FD_ERR_NOT_CONVERGED, "projected eigenproblem failed");
        auto tp2 = clk::now();
        t_rr += secs(tp0, tp1); t_eig += secs(tp1, tp2);
        nsel = std::min(nsel_max, m);
        theta.resize(nsel);
        Xr.assign((size_t)m * nsel, 0.0);
#pragma omp parallel for schedule(static) if (m >= 64)
        for (int jj = 0; jj < nsel; ++jj) {
            const int j = m - 1 - jj;
            theta[jj] = lam[j];
            for (int i = 0; i < m; ++i) {
                double corr = 0.0;
                for (int l = 0; l < m; ++l) corr += (S.G[i + (size_t)l * m_cap] - (i == l ? 1.0 : 0.0)) * U[l + (size_t)j * m];
                Xr[i + (size_t)jj * m] = U[i + (size_t)j * m] - 0.5 * corr;
            }
        }
        // ---- explicit residuals R_i = W x_i - theta_i Q x_i, into the spare panel -----------------
        // Leading pairs that converged with a margin at an earlier step are not re-evaluated every step (their Ritz
        // vectors only improve as the basis grows); before convergence is declared every pair is evaluated afresh.
        resid.resize(nsel, 1e300);
        const double thr = tol * std::fabs(theta[0]);
        bool all = false;
        int first = 0;                                             // X[:, i - first] holds the residual of pair i >= first
        double outside = 0.0;                                      // largest squared part of a wanted residual that the block ahead does not span
        for (int pass = 0; pass < 2; ++pass) {
            first = std::min(nlock, nsel);
            const int w = nsel - first;
            if (w > 0) {
                float* Sx = nullptr;
                const size_t cnt = (size_t)2 * m * w;
                FD_TRY(S.stage_slot(cnt, &Sx));
                for (int jj = 0; jj < w; ++jj)
                    for (int i = 0; i < m; ++i) {
                        const double x = Xr[i + (size_t)(first + jj) * m];
                        Sx[i + (size_t)jj * 2 * m] = (float)x;
                        Sx[m + i + (size_t)jj * 2 * m] = (float)(-theta[first + jj] * x);
                    }
                FD_TRY(S.send_slot(cnt));
                FD_TRY(nn_product(c, S.own(S.W, m, S.Q, m), S.d_S, 2 * m, w, S.X + r0, N, n));
                FD_TRY(col_sqnorms(c, S.X + r0, N, w, n, S.h));
                if (ahead > 0) FD_TRY(tn_product(c, S.own(S.R, ahead), S.own(S.X, w), n, S.h + w, S.d_scr, S.scr_n));
                FD_TRY(S.fetch(w + (int64_t)ahead * w));
                for (int jj = 0; jj < w; ++jj) resid[first + jj] = std::sqrt(std::max(0.0, S.h[jj]));
                outside = 0.0;
                for (int jj = 0; jj < w && first + jj < nwant && ahead > 0; ++jj) {
                    double rest = S.h[jj];
                    for (int i = 0; i < ahead; ++i) { const double z = S.h[w + i + (size_t)jj * ahead]; rest -= z * z; }
                    outside = std::max(outside, rest);
                }
            }
            nconv = 0;
            while (nconv < std::min(nwant, nsel) && resid[nconv] <= thr) ++nconv;
            all = nsel >= nwant;
            for (int i = 0; i < std::min(nwant, nsel); ++i) all = all && resid[i] <= thr;
            if (all && nlock > 0) { nlock = 0; continue; }       // verify the locked pairs before declaring convergence
            break;
        }
        {
            int lead = 0;
            while (lead < std::min(nwant, nsel) && resid[lead] <= 0.5 * thr) ++lead;
            nlock = lead;
        }
        auto tp3 = clk::now();
        t_res += secs(tp2, tp3);
        if (all) { final_status = FD_OK; break; }
        if (S.applies >= max_applies) break;
        int blocks = kMaxBlocks;                                  // blocks to append before the next Rayleigh-Ritz step
        {
            double worst = 0.0;
            for (int i = 0; i < std::min(nwant, nsel); ++i) worst = std::max(worst, resid[i]);
            if (nsel >= nwant) {
                if (worst < 0.9 * best_res) { best_res = worst; since_best = 0; }
                else since_best += S.applies - last_applies;
                // the worst residual's decay per product since the last step tells how many products are left
                if (last_worst > worst && worst > thr) {
                    last_rate = std::log(last_worst / worst) / std::max(1, S.applies - last_applies);
                    blocks = std::max(1, std::min(kMaxBlocks, (int)std::ceil(std::log(worst / thr) / last_rate)));
                }
                if (outside > kLost * kLost * worst * worst) krylov = false;
                last_worst = worst;
                last_applies = S.applies;
            }
            // the largest wanted residual has not improved by 10 % over 25 expansions and is within 2x of the target:
            // the operator's own rounding error is the floor; more applies do not help
            if (since_best >= 25 && best_res <= 2.0 * thr) break;
        }
        if (m >= N) break;                                        // basis spans everything: nothing more to add

        // ---- choose the expansion columns: wanted pairs above the tolerance first, then largest residuals first ---
        // (the buffer pairs' residuals are larger almost always; a wanted pair that the fp32 rounding of its residual holds
        // just above the tolerance would never be chosen; a small basis takes plain residual blocks throughout)
        std::vector<int> order(nsel);
        for (int i = 0; i < nsel; ++i) order[i] = i;
        std::sort(order.begin(), order.end(), [&](int a, int bb) {
            const bool wa = wanted_first && a < nwant && resid[a] > thr, wb = wanted_first && bb < nwant && resid[bb] > thr;
            return wa != wb ? wa : resid[a] > resid[bb];
        });
        const int want_new = (int)std::min<int64_t>(b, N - m);
        int p = ahead;
        if (ahead == 0) {
            std::vector<int> pick;
            for (int i = 0; i < nsel && (int)pick.size() < want_new; ++i)
                if (order[i] >= first && resid[order[i]] > 0.1 * thr) pick.push_back(order[i] - first);
            if (pick.empty()) { final_status = FD_OK; break; }
            p = (int)pick.size();
            krylov = krylov && p == b;
            FD_TRY(gather_cols(c, S.X + r0, S.R + r0, N, pick.data(), p, n));
        }

        // ---- thick restart when the new block would not fit ----------------------------------------
        if (m + p > m_cap) {
            int keep = std::max(nsel, kept_at(lam.data(), m));
            keep = std::min(keep, m_cap - p);
            keep = std::min(keep, m);
            // Ritz vectors for the kept block (beyond nsel use the uncorrected eigenvectors)
            float* Sk = nullptr;
            const size_t cnt = (size_t)m * keep;
            FD_TRY(S.stage_slot(cnt, &Sk));
            for (int jj = 0; jj < keep; ++jj) {
                const int j = m - 1 - jj;
                for (int i = 0; i < m; ++i)
                    Sk[i + (size_t)jj * m] = jj < nsel ? (float)Xr[i + (size_t)jj * m] : (float)U[i + (size_t)j * m];
            }
            FD_TRY(S.send_slot(cnt));
            FD_TRY(nn_product(c, S.own(S.Q, m), S.d_S, m, keep, S.X + r0, N, n));
            std::swap(S.Q, S.X);                                  // X now holds the old basis: reuse it for W
            FD_TRY(nn_product(c, S.own(S.W, m), S.d_S, m, keep, S.X + r0, N, n));
            std::swap(S.W, S.X);
            S.m = keep;
            ++S.restarts;
            if (!small_basis && since_best >= kStall && best_res <= 2.0 * thr && refreshes < kMaxRefreshes &&
                S.applies + (int)ceil_div(keep, b) < max_applies) {
                FD_TRY(S.apply_cols(0, keep, b));
                ++refreshes;
                since_best = 0; best_res = 1e300; last_worst = 0.0; nlock = 0;
            }
            // the kept columns are the Ritz vectors themselves (the loop may end below without another Rayleigh-Ritz step)
            Xr.assign((size_t)keep * nsel, 0.0);
            for (int jj = 0; jj < std::min(nsel, keep); ++jj) Xr[jj + (size_t)jj * keep] = 1.0;
            FD_TRY(S.full_projection());
        }
        auto tp4 = clk::now();
        t_restart += secs(tp3, tp4);
        // ---- append the residual block, then continue its Krylov space ---------------------------
        const double* z = nullptr;                                 // [Q B]^T B of the block to append, where it is known already
        int ldz = 0;
        std::vector<double> zkeep;
        const float* B = S.R;
        bool stuck = false;
        for (int blk = 0; blk < blocks; ++blk) {
            auto tb0 = clk::now();
            const bool have_image = ahead > 0;
            if (have_image) {
                FD_TRY(copy_cols(c, S.R + r0, N, S.Q + (int64_t)S.m * N + r0, N, p, n));
                FD_TRY(copy_cols(c, ahead_image + r0, N, S.W + (int64_t)S.m * N + r0, N, p, n));
                ahead = 0;
            } else FD_TRY(S.expand(B, p, z, ldz));
            krylov = krylov && p == b && (have_image || S.clean);
            if (p == 0) {
                if (blk > 0) break;                                // the continuation added nothing: back to the Ritz pairs
                // the residuals lie (numerically) inside the basis: try a random direction, give up after a few
                if (++stagnation > 3) { stuck = true; break; }
                p = (int)std::min<int64_t>(std::min(b, m_cap - S.m), N - S.m);
                FD_TRY(random_fill(c, S.R + r0, N, p, n, r0, 0xABCD1234u + (uint32_t)iter));
                FD_TRY(S.expand(S.R, p, nullptr, 0));
                if (p == 0) { stuck = true; break; }
            }
            auto tb1 = clk::now();
            t_orth += secs(tb0, tb1);
            if (!have_image) FD_TRY(S.apply_cols(S.m, p, b));
            auto tb2 = clk::now();
            FD_TRY(S.extend_projection(p));
            t_ext += secs(tb2, clk::now());
            if (S.applies >= max_applies || S.m + p > m_cap || S.m + p > N) break;
            // next block: M times this one; its projection [Q W_new]^T W_new was measured just now
            B = S.W + (int64_t)(S.m - p) * N;
            ldz = S.m + p;
            zkeep.assign(S.h + (size_t)p * ldz, S.h + (size_t)2 * p * ldz);
            z = zkeep.data();
        }
        if (stuck) break;
        // ---- the next block, ahead of the step that decides ----------------------------------------
        if (krylov && p == b && S.m + b <= N && S.applies + 1 < max_applies &&
            (nsel < nwant || last_worst * std::exp(-last_rate * (S.applies - last_applies)) > kAhead * tol * std::fabs(theta[0]))) {
            ldz = S.m + p;
            zkeep.assign(S.h + (size_t)p * ldz, S.h + (size_t)2 * p * ldz);
            FD_TRY(S.expand(S.W + (int64_t)(S.m - p) * N, p, zkeep.data(), ldz, S.R, S.X));
            krylov = p == b && S.clean;
            if (p > 0) FD_TRY(S.apply_block(S.R, ahead_image, p, b));
            ahead = p;
        }
    }

    // ---- outputs: evecs = Q X[:, 0 : k + 1) ----------------------------------------------------------
    const int nout = std::min(nwant, nsel);
    {
        const int m = S.m;
        float* Sx = nullptr;
        const size_t cnt = (size_t)m * nout;
        FD_TRY(S.stage_slot(cnt, &Sx));
        for (size_t i = 0; i < cnt; ++i) Sx[i] = (float)Xr[i];
        FD_TRY(S.send_slot(cnt));
        FD_TRY(nn_product(c, S.own(S.Q, m), S.d_S, m, nout, evecs_dev + r0, ldv, n));
        FD_TRY(gather_rows(c, evecs_dev, ldv, nout));              // complete eigenvectors on every rank
        for (int i = 0; i < nwant; ++i) evals_host[i] = i < nout ? theta[i] : 0.0;
        FD_CUDA(c, cudaStreamSynchronize(c->stream));
    }
#ifdef FD_EIGS_TIMING
    fprintf(stderr, "fd_eigs: staging init %.3f s, total so far %.3f s\n", t_init, secs(t_start, clk::now()));
    fprintf(stderr, "fd_eigs: RR setup %.3f s, small eig %.3f s, residuals %.3f s, select+restart %.3f s, orthogonalise %.3f s, applies on the GPU %.3f s, wait for them and extend projection %.3f s\n",
            t_rr, t_eig, t_res, t_restart, t_orth, S.t_apply, t_ext);
#else
    (void)t_init; (void)t_rr; (void)t_eig; (void)t_res; (void)t_restart; (void)t_orth; (void)t_ext;
#endif
    if (info) {
        info->applies = S.applies; info->restarts = S.restarts; info->converged = nconv; info->basis_cols = S.m;
        double mx = 0.0;
        for (int i = 0; i < nout; ++i) mx = std::max(mx, resid[i]);
        info->max_residual = mx;
        info->seconds_apply = S.t_apply;
        info->seconds_total = secs(t_start, clk::now());
    }
    if (final_status != FD_OK) return fail(c, FD_ERR_NOT_CONVERGED, "fd_eigs: %d of %d pairs converged after %d applies", nconv, nwant, S.applies);
    return FD_OK;
}
