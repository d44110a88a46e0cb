// FP64 dense helpers (internal): GEMM and symmetric eigensolver.
#pragma once
#include <vector>
#include <algorithm>

#include "common.cuh"

namespace caspt2 {

// Optional device-time accounting for one kernel (CUDA events on the launching stream).
struct KernelTimer {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  double ms = 0.0;       // summed device time
  double flops = 0.0;    // summed algorithmic flops
  double bytes = 0.0;    // summed algorithmic DRAM bytes
  long launches = 0;
  // the panel launches of the blocked reduction alone (k_latrd): an event pair per launch
  // (grown on demand, owned by the timer's holder), device time and the bytes of the
  // trailing matrix its matrix-vector products read (8 n1^2 per column)
  std::vector<cudaEvent_t> pev;
  double pms = 0.0, pbytes = 0.0;
  long plaunches = 0;
};

// Optional record of the FP64 GEMM launches of one host thread: an event pair around each
// launch (device time) and its algorithmic flops (2 M N K; the symmetric-output form its
// computed tiles).  Up to kGemmTimerPairs launches per collection; later ones run untimed.
constexpr int kGemmTimerPairs = 4096;
struct GemmTimer {
  cudaEvent_t ev[2 * kGemmTimerPairs] = {};
  double flops[kGemmTimerPairs] = {};
  int used = 0;
  bool ready = false;
};
cudaError_t gemm_timer_init(GemmTimer& t);
void gemm_timer_release(GemmTimer& t);
void set_gemm_timer(GemmTimer* t);   // this thread's dgemm launches are recorded (nullptr: off)
// Sum of the recorded launches (call after the stream has synchronised); resets the record.
cudaError_t gemm_timer_collect(GemmTimer& t, double* ms, double* flops, long* launches);

// Row-major C = alpha * op(A) op(B) + beta * C, op = transpose when the flag is set.
// Batched over `batch` with element strides sA, sB, sC.
cudaError_t dgemm(int M, int N, int K, double alpha, const double* A, int lda, bool ta,
                  const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                  cudaStream_t s, int batch = 1, long sA = 0, long sB = 0, long sC = 0);
// C[i][j] (ldc) = alpha * sum_k A(i, k) B(j, k) + beta * C, with general strides and K in runs:
// A(i, k) = A[i * ars + (k / akin) * akout + (k % akin) * acs], B alike.
struct KView { const double* X; long rs, cs, kin, kout; };
// sym: the result is known to be symmetric (M = N, beta = 0), half of its tiles are formed.
cudaError_t dgemm_views(int M, int N, int K, double alpha, const KView& A, const KView& B,
                        double beta, double* C, long ldc, cudaStream_t s, bool sym = false);
// Same product when the N x N result is known to be symmetric (A^T A, X^T F X): only the
// upper-triangle tiles are computed, each written to both triangles.
cudaError_t dgemm_sym(int N, int K, double alpha, const double* A, int lda, bool ta,
                      const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                      cudaStream_t s);

// Eigenpairs of a symmetric m x m matrix by Householder tridiagonalisation, eigenvalues,
// inverse iteration and back-transformation (eig_tridiag.cu).  A is destroyed; w[m]
// ascending; V[m][m] eigenvectors as columns.  work >= sym_eig_tridiag_work(m) doubles.
size_t sym_eig_tridiag_work(int m);
// oz (optional, on): the Newton-Schulz correction Z (1/2)(I - Z^T Z), a term of the size of
// the orthogonality error, runs as a split-BF16 product with just enough slices.
struct OzWork;
// nkept (optional): only the vectors of the eigenvalues >= wmin are formed, V is m x *nkept
// (ascending), and *nkept is known on the host when the call returns.
int sym_eig_tridiag(double* A, int m, double* w, double* V, double* work, cudaStream_t s,
                    KernelTimer* tm = nullptr, OzWork* oz = nullptr, double wmin = 0.0,
                    int* nkept = nullptr);

// The same in one block in shared memory, m <= kSectorBlockMax (sector_block.cu): V is m x m,
// or m x *nkept with nkept.  work >= sym_eig_work(m).  Synchronises the stream.
int sym_eig_block(const double* A, int m, double* w, double* V, double* work, cudaStream_t s,
                  double wmin = -1e300, int* nkept = nullptr);

// Eigenpairs of A (destroyed): w[m] ascending, V[m][m] eigenvectors as columns.  One block for
// up to kSectorBlockMax rows, the whole GPU above.  A single matrix takes one block 0.4 ms at 33 rows,
// 1.0 at 64 and 2.0 at 96, the large path 0.34, 0.64 and 0.86; the line stays at the size of
// the sectors' solver, which leaves residuals of 1e-14 of the norm and vectors orthogonal to
// 1e-14 for repeated eigenvalues too (polish), the large path up to 1e-12 and 1e-13.
int sym_eig(double* A, int m, double* w, double* V, double* work, cudaStream_t s,
            KernelTimer* tm = nullptr, OzWork* oz = nullptr);
inline size_t sym_eig_work(int m) {
  return std::max<size_t>((size_t)5 * m * m + 2 * m + 64, sym_eig_tridiag_work(m));
}

// Eigenvalues w[m] (all) and the eigenvectors of those >= wmin: V is m x *nkept (ascending).
// The vectors below the cut are not formed: an overlap matrix of rank r spends its inverse
// iteration, cluster orthogonalisation and back-transformation on r columns, and its null
// space (one cluster of equal eigenvalues, serial in the Gram-Schmidt: 0.9 s of the 1.3 s of
// a c42 a6 v350 n4 solve) costs nothing.
int sym_eig_above(double* A, int m, double wmin, double* w, double* V, int* nkept, double* work,
                  cudaStream_t s, KernelTimer* tm = nullptr, OzWork* oz = nullptr);

}  // namespace caspt2
