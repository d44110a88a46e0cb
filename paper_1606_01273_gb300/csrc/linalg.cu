// FP64 dense building blocks: tiled GEMMs, and the choice of the symmetric eigensolver.
#include "linalg.cuh"
#include "sector_block.cuh"

namespace caspt2 {

// C[i][j] = alpha * sum_k A(i,k) B(k,j) + beta * C[i][j]
// A(i,k) = ta ? A[k*lda + i] : A[i*lda + k]; B(k,j) = tb ? B[j*ldb + k] : B[k*ldb + j]
constexpr int kGT = 64, kGK = 16;
__global__ void __launch_bounds__(256)
k_dgemm(int M, int N, int K, double alpha, const double* __restrict__ A, int lda, int ta,
        const double* __restrict__ B, int ldb, int tb, double beta, double* __restrict__ C, int ldc,
        long sA, long sB, long sC, int sym) {
  __shared__ double sa[kGK][kGT + 1], sb[kGK][kGT + 1];
  A += blockIdx.z * sA;
  B += blockIdx.z * sB;
  C += blockIdx.z * sC;
  int by = blockIdx.y, bx = blockIdx.x;
  if (sym) {          // symmetric result: upper-triangle tiles only, blockIdx.x linear
    const int T = (N + kGT - 1) / kGT;
    int rem = blockIdx.x;
    by = 0;
    while (rem >= T - by) { rem -= T - by; ++by; }
    bx = by + rem;
  }
  const int i0 = by * kGT, j0 = bx * kGT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += kGK) {
    for (int l = threadIdx.x; l < kGK * kGT; l += 256) {
      int kk, ii;
      if (ta) { ii = l % kGT; kk = l / kGT; } else { kk = l % kGK; ii = l / kGK; }
      const int gi = i0 + ii, gk = k0 + kk;
      double v = 0.0;
      if (gi < M && gk < K) v = ta ? A[(long)gk * lda + gi] : A[(long)gi * lda + gk];
      sa[kk][ii] = v;
    }
    for (int l = threadIdx.x; l < kGK * kGT; l += 256) {
      int kk, jj;
      if (tb) { kk = l % kGK; jj = l / kGK; } else { jj = l % kGT; kk = l / kGT; }
      const int gj = j0 + jj, gk = k0 + kk;
      double v = 0.0;
      if (gj < N && gk < K) v = tb ? B[(long)gj * ldb + gk] : B[(long)gk * ldb + gj];
      sb[kk][jj] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kGK; ++kk) {
      double ra[4], rb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { ra[q] = sa[kk][ty + 16 * q]; rb[q] = sb[kk][tx + 16 * q]; }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma(ra[p], rb[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gi = i0 + ty + 16 * p, gj = j0 + tx + 16 * q;
      if (gi < M && gj < N) {
        double* c = C + (long)gi * ldc + gj;
        *c = alpha * acc[p][q] + (beta == 0.0 ? 0.0 : beta * *c);
        if (sym && bx != by) {
          double* ct = C + (long)gj * ldc + gi;
          *ct = alpha * acc[p][q] + (beta == 0.0 ? 0.0 : beta * *ct);
        }
      }
    }
}

// Small-tile variant for products with a short edge: a TM x TN tile (each <= 32,
// fitted to M and N) per block, up to 4 outputs per thread, K in chunks of 8.
constexpr int kST = 32, kSK = 8;
__global__ void __launch_bounds__(256)
k_dgemm_s(int M, int N, int K, double alpha, const double* __restrict__ A, int lda, int ta,
          const double* __restrict__ B, int ldb, int tb, double beta, double* __restrict__ C,
          int ldc, int TM, int TN, int tn, long sA, long sB, long sC) {
  __shared__ double sa[kSK][kST + 1], sb[kSK][kST + 1];
  A += blockIdx.y * sA;
  B += blockIdx.y * sB;
  C += blockIdx.y * sC;
  const int i0 = (int)(blockIdx.x / tn) * TM, j0 = (int)(blockIdx.x % tn) * TN;
  const int nout = TM * TN;
  int oi[4], oj[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int q = threadIdx.x + 256 * r;
    oi[r] = q < nout ? q / TN : 0;
    oj[r] = q < nout ? q % TN : 0;
  }
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int k0 = 0; k0 < K; k0 += kSK) {
    for (int l = threadIdx.x; l < kSK * TM; l += 256) {
      int kk, ii;
      if (ta) { ii = l % TM; kk = l / TM; } else { kk = l % kSK; ii = l / kSK; }
      const int gi = i0 + ii, gk = k0 + kk;
      double v = 0.0;
      if (gi < M && gk < K) v = ta ? A[(long)gk * lda + gi] : A[(long)gi * lda + gk];
      sa[kk][ii] = v;
    }
    for (int l = threadIdx.x; l < kSK * TN; l += 256) {
      int kk, jj;
      if (tb) { kk = l % kSK; jj = l / kSK; } else { jj = l % TN; kk = l / TN; }
      const int gj = j0 + jj, gk = k0 + kk;
      double v = 0.0;
      if (gj < N && gk < K) v = tb ? B[(long)gj * ldb + gk] : B[(long)gk * ldb + gj];
      sb[kk][jj] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kSK; ++kk) {
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[r] = fma(sa[kk][oi[r]], sb[kk][oj[r]], acc[r]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int q = threadIdx.x + 256 * r;
    const int gi = i0 + oi[r], gj = j0 + oj[r];
    if (q < nout && gi < M && gj < N) {
      double* c = C + (long)gi * ldc + gj;
      *c = alpha * acc[r] + (beta == 0.0 ? 0.0 : beta * *c);
    }
  }
}

namespace {
thread_local GemmTimer* tl_gemm_timer = nullptr;

// Start of a timed launch: the slot of its event pair, or -1.
int gemm_timer_begin(cudaStream_t s) {
  GemmTimer* t = tl_gemm_timer;
  if (!t || !t->ready || t->used >= kGemmTimerPairs) return -1;
  const int slot = t->used++;
  cudaEventRecord(t->ev[2 * slot], s);
  return slot;
}
void gemm_timer_end(int slot, double flops, cudaStream_t s) {
  if (slot < 0) return;
  GemmTimer* t = tl_gemm_timer;
  cudaEventRecord(t->ev[2 * slot + 1], s);
  t->flops[slot] = flops;
}
}  // namespace

cudaError_t gemm_timer_init(GemmTimer& t) {
  if (t.ready) return cudaSuccess;
  for (auto& e : t.ev) {
    const cudaError_t r = cudaEventCreate(&e);
    if (r != cudaSuccess) return r;
  }
  t.used = 0;
  t.ready = true;
  return cudaSuccess;
}

void gemm_timer_release(GemmTimer& t) {
  for (auto& e : t.ev)
    if (e) cudaEventDestroy(e);
  t.ready = false;
}

void set_gemm_timer(GemmTimer* t) { tl_gemm_timer = t; }

cudaError_t gemm_timer_collect(GemmTimer& t, double* ms, double* flops, long* launches) {
  double tot = 0.0, fl = 0.0;
  for (int k = 0; k < t.used; ++k) {
    float x = 0.f;
    const cudaError_t r = cudaEventElapsedTime(&x, t.ev[2 * k], t.ev[2 * k + 1]);
    if (r != cudaSuccess) return r;
    tot += x;
    fl += t.flops[k];
  }
  *ms = tot;
  *flops = fl;
  *launches = t.used;
  t.used = 0;
  return cudaSuccess;
}

cudaError_t dgemm(int M, int N, int K, double alpha, const double* A, int lda, bool ta,
                  const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                  cudaStream_t s, int batch, long sA, long sB, long sC) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  const int slot = gemm_timer_begin(s);
  // padded work of the 64 x 64 tiles against tiles fitted to M and N (<= 32)
  const double pad64 = (double)((M + kGT - 1) / kGT * kGT) * ((N + kGT - 1) / kGT * kGT) /
                       ((double)M * N);
  ++launch_counter();
  if (pad64 > 1.3 || (M + kGT - 1) / kGT > 65535) {
    const int tm = (M + kST - 1) / kST, tn = (N + kST - 1) / kST;
    const int TM = (M + tm - 1) / tm, TN = (N + tn - 1) / tn;
    dim3 grid((unsigned)((long)tm * tn), batch);
    k_dgemm_s<<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C,
                                   ldc, TM, TN, tn, sA, sB, sC);
  } else {
    dim3 grid((N + kGT - 1) / kGT, (M + kGT - 1) / kGT, batch);
    k_dgemm<<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C,
                                 ldc, sA, sB, sC, 0);
  }
  gemm_timer_end(slot, 2.0 * M * N * (double)K * batch, s);
  return cudaGetLastError();
}

cudaError_t dgemm_sym(int N, int K, double alpha, const double* A, int lda, bool ta,
                      const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                      cudaStream_t s) {
  const int T = (N + kGT - 1) / kGT;
  const double pad64 = (double)T * kGT * T * kGT / ((double)N * N);
  if (N <= 0 || pad64 > 1.3 || T > 2048)
    return dgemm(N, N, K, alpha, A, lda, ta, B, ldb, tb, beta, C, ldc, s);
  ++launch_counter();
  const int slot = gemm_timer_begin(s);
  dim3 grid((unsigned)((long)T * (T + 1) / 2), 1, 1);
  k_dgemm<<<grid, 256, 0, s>>>(N, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C,
                               ldc, 0, 0, 0, 1);
  gemm_timer_end(slot, 2.0 * kGT * kGT * (double)K * ((double)T * (T + 1) / 2), s);
  return cudaGetLastError();
}

int sym_eig_above(double* A, int m, double wmin, double* w, double* V, int* nkept, double* work,
                  cudaStream_t s, KernelTimer* tm, OzWork* oz) {
  *nkept = 0;
  if (m <= 0) return CASPT2_OK;
  return m <= kSectorBlockMax ? sym_eig_block(A, m, w, V, work, s, wmin, nkept)
                              : sym_eig_tridiag(A, m, w, V, work, s, tm, oz, wmin, nkept);
}

int sym_eig(double* A, int m, double* w, double* V, double* work, cudaStream_t s,
            KernelTimer* tm, OzWork* oz) {
  if (m <= 0) return CASPT2_OK;
  return m <= kSectorBlockMax ? sym_eig_block(A, m, w, V, work, s)
                              : sym_eig_tridiag(A, m, w, V, work, s, tm, oz);
}

}  // namespace caspt2
