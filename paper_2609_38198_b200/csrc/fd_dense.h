// Tall-skinny dense helpers (fd_dense.cu) and the host symmetric eigensolver (fd_symeig.cpp).
#pragma once
#include <functional>
#include <vector>

#include "fd_internal.h"

namespace fd {

// Columns of a tall matrix: m1 columns at p1 followed by m2 columns at p2 (m2 may be 0), column pitch ld.
struct Panel { const float* p1; int m1; const float* p2; int m2; int64_t ld; };
inline Panel panel(const float* p, int m, int64_t ld) { return Panel{p, m, nullptr, 0, ld}; }
inline Panel panel(const float* p1, int m1, const float* p2, int m2, int64_t ld) { return Panel{p1, m1, p2, m2, ld}; }

// out[(A columns) x (B columns)] (column-major doubles; device or page-locked host memory) = A^T B over N rows, fp64 accumulation.
// scratch: device doubles for the per-chunk partials.
fd_status tn_product(fd_ctx* c, const Panel& A, const Panel& B, int64_t N, double* out, double* scratch, size_t scratch_doubles);
// C[N x p] = A[N x m] S[m x p]; S_dev column-major floats with pitch lds.  C must not alias A.
fd_status nn_product(fd_ctx* c, const Panel& A, const float* S_dev, int lds, int p, float* C, int64_t ldc, int64_t N);
// dst[:, i] = src[:, idx[i]] for p <= 256 columns, both with column pitch ld.
fd_status gather_cols(fd_ctx* c, const float* src, float* dst, int64_t ld, const int* idx, int p, int64_t N);
// out[c] = |A[:, c]|^2 (fp64; device or page-locked host memory) for the first p columns.
fd_status col_sqnorms(fd_ctx* c, const float* A, int64_t lda, int p, int64_t N, double* out);
// Counter-based uniform(-1, 1) fill of N rows x p columns; row i of A is row row0 + i of the stream, so a row range of
// a larger block gets the values the whole block would.
fd_status random_fill(fd_ctx* c, float* A, int64_t lda, int p, int64_t N, int64_t row0, uint32_t seed);
fd_status sqrt_vec(fd_ctx* c, const float* d, float* out, int64_t N);
fd_status copy_cols(fd_ctx* c, const float* src, int64_t lds, float* dst, int64_t ldd, int p, int64_t N);

// y += a x, and x . y, on the host (fd_symeig.cpp: with the widest vectors the machine has).
void host_axpy(double* y, const double* x, double a, int n);
double host_dot(const double* x, const double* y, int n);

// Eigen-decomposition of a dense symmetric n x n matrix (column-major, only read).  On return evals ascending (all n) and
// evecs n x n column-major with orthonormal columns; with 0 <= nvec < n only the columns of the nvec LARGEST eigenvalues
// (columns n - nvec .. n - 1) are computed, the others are zero.  Householder tridiagonalisation followed by implicit
// symmetric QR.  Returns false if the iteration fails to converge.  needed, if given, says how many of the nvec columns are needed
// once the (ascending) eigenvalues are known.
bool sym_eig(const double* A, int n, std::vector<double>& evals, std::vector<double>& evecs, int nvec = -1,
             const std::function<int(const double*)>& needed = nullptr);

}  // namespace fd
