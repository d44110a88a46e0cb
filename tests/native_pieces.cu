// C entry points to single pieces of the library for the tests: host arrays in, host arrays out.
#include <cuda_runtime.h>

#include "../paper_1606_01273_gb300/csrc/linalg.cuh"

namespace {

__global__ void k_recip(const double* x, long n, double* y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = caspt2::recip(x[i]);
}

__global__ void k_root(const double* x, long n, double* r, double* ir) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    caspt2::root_and_recip(x[i], r[i], ir[i]);
}

struct Dev {
  double* p = nullptr;
  explicit Dev(size_t n) { if (cudaMalloc(&p, (n ? n : 1) * sizeof(double)) != cudaSuccess) p = nullptr; }
  ~Dev() { cudaFree(p); }
};

}  // namespace

extern "C" {

int np_recip(const double* x, long n, double* y) {
  Dev dx(n), dy(n);
  if (!dx.p || !dy.p) return CASPT2_ENOMEM;
  CASPT2_CUDA_TRY(cudaMemcpy(dx.p, x, n * sizeof(double), cudaMemcpyHostToDevice));
  k_recip<<<152, 256>>>(dx.p, n, dy.p);
  CASPT2_CUDA_TRY(cudaGetLastError());
  CASPT2_CUDA_TRY(cudaMemcpy(y, dy.p, n * sizeof(double), cudaMemcpyDeviceToHost));
  return CASPT2_OK;
}

int np_root(const double* x, long n, double* r, double* ir) {
  Dev dx(n), dr(n), di(n);
  if (!dx.p || !dr.p || !di.p) return CASPT2_ENOMEM;
  CASPT2_CUDA_TRY(cudaMemcpy(dx.p, x, n * sizeof(double), cudaMemcpyHostToDevice));
  k_root<<<152, 256>>>(dx.p, n, dr.p, di.p);
  CASPT2_CUDA_TRY(cudaGetLastError());
  CASPT2_CUDA_TRY(cudaMemcpy(r, dr.p, n * sizeof(double), cudaMemcpyDeviceToHost));
  CASPT2_CUDA_TRY(cudaMemcpy(ir, di.p, n * sizeof(double), cudaMemcpyDeviceToHost));
  return CASPT2_OK;
}

// Eigenvalues w [m] and the vectors V [m][*nk] of those at or above wmin; block: in the one-block
// solver, else by the library's choice.
int np_eig_above(const double* A, int m, double wmin, double* w, double* V, int* nk, int block) {
  const size_t mm = (size_t)m * m;
  Dev dA(mm), dw(m), dV(mm), work(caspt2::sym_eig_work(m));
  if (!dA.p || !dw.p || !dV.p || !work.p) return CASPT2_ENOMEM;
  CASPT2_CUDA_TRY(cudaMemcpy(dA.p, A, mm * sizeof(double), cudaMemcpyHostToDevice));
  const int st = block ? caspt2::sym_eig_block(dA.p, m, dw.p, dV.p, work.p, nullptr, wmin, nk)
                       : caspt2::sym_eig_above(dA.p, m, wmin, dw.p, dV.p, nk, work.p, nullptr);
  if (st != CASPT2_OK) return st;
  CASPT2_CUDA_TRY(cudaMemcpy(w, dw.p, m * sizeof(double), cudaMemcpyDeviceToHost));
  CASPT2_CUDA_TRY(cudaMemcpy(V, dV.p, (size_t)m * *nk * sizeof(double), cudaMemcpyDeviceToHost));
  return CASPT2_OK;
}

}  // extern "C"
