// Eigenbases of the small sectors of classes A-G, every sector of a solve in one launch.
//
// One block solves one sector (msec <= kSectorBlockMax rows): overlap S and active Fock F from
// the class matrices, S = Q s Q^T, X = Q s^(-1/2) over s >= thresh (Sec. II.B), X^T F X =
// P diag(omega) P^T, Y = X P.  Both eigenproblems run in shared memory: Householder
// tridiagonalisation, eigenvalues (single-precision multisection, then a safeguarded secant
// on the last principal minor in FP64), inverse iteration, Gram-Schmidt, back-transformation.
//
// What bounds it: the FP64 unit of an SM sub-partition takes one warp instruction in 64
// clocks and answers after 68, so a sector is a chain of about 25 dependent FP64
// instructions a row and stage, whatever the thread count; the way to more work a second is
// more sectors side by side, and a solve has 11 (MS-MR) to 11 n (SS-SR) of them.  The
// stages avoid FP64 instructions that other units can do (comparisons on bit patterns, the
// first 17 bits of every eigenvalue in single precision) and block-wide reductions (one warp
// reduces, the others wait).
#include <algorithm>
#include <vector>

#include "class_ag.cuh"
#include "class_dev.cuh"
#include "eig_dev.cuh"
#include "linalg.cuh"
#include "sector_block.cuh"

namespace caspt2 {

namespace {

constexpr int kNT = 256;                       // threads of a sector's block
constexpr int kNW = kNT / 32;

// Shared vectors of the eigenproblem, m doubles each, after the two m x m matrices.
struct Vecs {
  double *d, *e, *e2, *tau, *w, *u, *p, *lo, *hi;
  float *df, *ef;
};
constexpr int kNVec = 11;                      // d .. hi, and the two float copies in one

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 2^e, -1022 <= e <= 1023
__device__ __forceinline__ double exp2i(int e) {
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// Householder reduction of the symmetric A (rows of stride ld): d, e, and the reflectors
// H_k = 1 - tau_k u u^T with u in row k right of the diagonal (not normalised:
// u = x + sign(x_0) |x| e_0, tau = 1 / (|x| (|x| + |x_0|))).
__device__ void tridiagonalise(double* A, int ld, int m, const Vecs& q) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = 0; k + 2 < m; ++k) {
    const int n1 = m - k - 1;
    double* x = A + k * ld + k + 1;
    if (warp == 0) {
      double s = 0.0;
      for (int j = lane + 1; j < n1; j += 32) s = fma(x[j], x[j], s);
      s = warp_sum(s);
      const double al = x[0];
      const double sig = fma(al, al, s);
      double beta = al, t = 0.0, u0 = al;
      if (s != 0.0 && sig > 1e-280) {
        const double nr = sqrt(sig);
        beta = -copysign(nr, al);
        u0 = al - beta;
        t = 1.0 / (nr * (nr + fabs(al)));
      }
      __syncwarp();
      for (int j = lane; j < n1; j += 32) q.u[j] = j == 0 ? u0 : x[j];
      if (lane == 0) {
        x[0] = u0;
        q.tau[k] = t;
        q.d[k] = A[k * ld + k];
        q.e[k] = beta;
      }
    }
    __syncthreads();
    // p = A22 u: eight lanes a row
    {
      const int sub = lane & 7;
      for (int i0 = 0; i0 < n1; i0 += kNT / 8) {
        const int i = i0 + (threadIdx.x >> 3);
        double s0 = 0.0, s1 = 0.0;
        if (i < n1) {
          const double* row = A + (k + 1 + i) * ld + k + 1;
          int j = sub;
          for (; j + 8 < n1; j += 16) {
            s0 = fma(row[j], q.u[j], s0);
            s1 = fma(row[j + 8], q.u[j + 8], s1);
          }
          if (j < n1) s0 = fma(row[j], q.u[j], s0);
        }
        if (i0 + warp * 4 < n1) {              // whole warps only
          double s = s0 + s1;
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (sub == 0 && i < n1) q.p[i] = s;
        }
      }
    }
    __syncthreads();
    // w = tau p - (tau^2 / 2)(u . p) u, in place of p.  A sector without overlap is rounding
    // noise that shrinks by 1e-17 a step: tau reaches 1e280 and tau^2 leaves the FP64 range,
    // tau (u . p), of the size of A22, does not.
    if (warp == 0) {
      double s = 0.0;
      for (int j = lane; j < n1; j += 32) s = fma(q.u[j], q.p[j], s);
      s = warp_sum(s);
      const double t = q.tau[k], ts = t * s, g = 0.5 * t * ts;
      for (int j = lane; j < n1; j += 32) q.p[j] = fma(-g, q.u[j], t * q.p[j]);
    }
    __syncthreads();
    // A22 -= u w^T + w u^T: 32-column chunks from the diagonal's on, the rest mirrored
    for (int i = warp; i < n1; i += kNW) {
      const double ui = q.u[i], wi = q.p[i];
      double* row = A + (k + 1 + i) * ld + k + 1;
      const int c0 = i & ~31;
      for (int j = c0 + lane; j < n1; j += 32) {
        const double v = fma(-wi, q.u[j], fma(-ui, q.p[j], row[j]));
        row[j] = v;
        if (j - lane != c0) A[(k + 1 + j) * ld + k + 1 + i] = v;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (m >= 2) {
      q.d[m - 2] = A[(m - 2) * ld + m - 2];
      q.e[m - 2] = A[(m - 2) * ld + m - 1];
    }
    q.d[m - 1] = A[(m - 1) * ld + m - 1];
    q.e[m - 1] = 0.0;
  }
  __syncthreads();
}

// C[i * N + j] = sum_k A[i * ai + k * ak] B[k * bk + j * bj], two outputs a thread in flight.
__device__ void block_mm(int M, int N, int K, const double* A, int ai, int ak, const double* B,
                         int bk, int bj, double* C) {
  const int total = M * N;
  for (int o = threadIdx.x; o < total; o += 2 * kNT) {
    const int o2 = o + kNT < total ? o + kNT : o;
    const double *a0 = A + (o / N) * ai, *b0 = B + (o % N) * bj;
    const double *a1 = A + (o2 / N) * ai, *b1 = B + (o2 % N) * bj;
    double s0 = 0.0, s1 = 0.0;
    for (int k = 0; k < K; ++k) {
      s0 = fma(a0[k * ak], b0[k * bk], s0);
      s1 = fma(a1[k * ak], b1[k * bk], s1);
    }
    C[o] = s0;
    if (o2 != o) C[o2] = s1;
  }
}

// Eigenvectors Z [m][nc] of T to the residual's second order: z_j += sum_i z_i (z_i . r_j) / (w_j -
// w_i), r_j = T z_j - w_j z_j, as rotations of pairs (orthogonality stays).  The vectors of equal
// eigenvalues come from independent starts; one that Gram-Schmidt leaves little of carries its
// rounding that much enlarged, and the vectors orthogonalised against it with it (4e-13 at 64 rows
// with 26 equal eigenvalues, where a Jacobi sweep reaches 1e-15).  Pairs closer than 1e7 times the
// residual stay as they are.  Without such a residual, the usual case, only r is formed.
// scr: 3 m nc doubles.
__device__ void polish(int m, int nc, double tn, const double* wk, double* Z, double* scr,
                       const Vecs& q) {
  const unsigned long long lim = abits(1e-14 * tn);
  bool bad = false;
  for (int t = threadIdx.x; t < m * nc; t += kNT) {
    const int i = t / nc, j = t % nc;
    double r = (q.d[i] - wk[j]) * Z[t];
    if (i > 0) r = fma(q.e[i - 1], Z[t - nc], r);
    if (i + 1 < m) r = fma(q.e[i], Z[t + nc], r);
    scr[t] = r;
    bad = bad || abits(r) > lim;
  }
  if (!__syncthreads_or(bad)) return;
  double *E = scr + (long)m * nc, *dZ = E + (long)m * nc;
  block_mm(nc, nc, m, Z, 1, nc, scr, nc, 1, E);
  __syncthreads();
  for (int t = threadIdx.x; t < nc * nc; t += kNT) {       // the pair (i < j) by one thread
    const int i = t / nc, j = t % nc;
    if (i > j) continue;
    const double g = wk[j] - wk[i], e = 0.5 * (E[i * nc + j] + E[j * nc + i]);
    const double c = i < j && fabs(e) < 1e-7 * g ? e / g : 0.0;
    E[i * nc + j] = c;
    E[j * nc + i] = -c;
  }
  __syncthreads();
  block_mm(m, nc, nc, Z, nc, 1, E, nc, 1, dZ);
  __syncthreads();
  for (int t = threadIdx.x; t < m * nc; t += kNT) Z[t] += dZ[t];
  __syncthreads();
}

// Eigenpairs of A (destroyed; stride ld): q.w holds all m eigenvalues ascending, Z [m][nc] the
// vectors of the last nc, of which the last nk have eigenvalues >= wmin (eig_guard).  scr: 4 m
// nc doubles and m nc bytes.  Returns nk, or -1 when the matrix holds a NaN or an infinity.
// T is scaled by a power of two to a norm in [1, 2): the brackets' widths and the ranges of the
// recurrences are then relative to the norm (a sector of weakly occupied orbitals has a norm of
// 1e-6 and keeps all its digits), and no rounding changes.
__device__ int eig_block(double* A, int ld, int m, double wmin, double* Z, double* scr,
                         const Vecs& q, double* sh, int& nc) {
  nc = 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  tridiagonalise(A, ld, m, q);
  // Gershgorin interval
  if (warp == 0) {
    double glo = 1e300, ghi = -1e300, tn = 0.0;
    bool bad = false;
    for (int i = lane; i < m; i += 32) {
      const double r = (i > 0 ? fabs(q.e[i - 1]) : 0.0) + (i < m - 1 ? fabs(q.e[i]) : 0.0);
      glo = fmin(glo, q.d[i] - r);
      ghi = fmax(ghi, q.d[i] + r);
      tn = fmax(tn, fabs(q.d[i]) + r);
      bad = bad || !(fabs(q.d[i]) + r < 1e300);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
      ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
      tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    }
    bad = __any_sync(0xffffffffu, bad);
    const int ex = tn > 0x1p-1000 ? (int)(abits(tn) >> 52) - 1023 : 0;
    const double sc = exp2i(-ex);
    __syncwarp();
    for (int i = lane; i < m; i += 32) {
      const double di = q.d[i] * sc, ei = q.e[i] * sc;
      q.d[i] = di;
      q.e[i] = ei;
      q.e2[i] = ei * ei;
      q.df[i] = (float)di;
      q.ef[i] = (float)(ei * ei);
    }
    if (lane == 0) {
      tn *= sc;
      const double pad = 2.2e-16 * tn * 4.0;
      sh[0] = glo * sc - pad;
      sh[1] = ghi * sc + pad;
      sh[2] = tn;
      sh[3] = bad ? 1.0 : 0.0;
      sh[6] = sc;
      sh[7] = exp2i(ex);
    }
  }
  __syncthreads();
  if (sh[3] != 0.0) return -1;
  const double glo = sh[0], ghi = sh[1], tn = sh[2], unscale = sh[7];
  wmin *= sh[6];
  // single-precision brackets, eight lanes an eigenvalue; then FP64, one lane each
  for (int j0 = 0; j0 < m; j0 += kNT / 8) {
    const int j = j0 + (threadIdx.x >> 3);
    float flo, fhi;
    bisect_f32(q.df, q.ef, m, min(j, m - 1), glo, ghi, flo, fhi);
    if (j < m && (threadIdx.x & 7) == 0) {
      q.lo[j] = flo;
      q.hi[j] = fhi;
    }
  }
  __syncthreads();
  const double tol = kEigTol * tn;
  for (int j = threadIdx.x; j < m; j += kNT)
    q.w[j] = eigenvalue_f64(q.d, q.e2, m, j, glo, ghi, q.lo[j], q.hi[j], tol,
                             eig_guard(wmin, tn));
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    while (c < m && q.w[c] < wmin) ++c;
    sh[4] = (double)(m - c);
    if (c < m)
      while (c > 0 && q.w[c - 1] >= eig_guard(wmin, tn)) --c;
    sh[5] = (double)(m - c);
  }
  __syncthreads();
  const int nk = (int)sh[4];
  nc = (int)sh[5];
  if (nk == 0) {
    for (int j = threadIdx.x; j < m; j += kNT) q.w[j] *= unscale;
    __syncthreads();
    return 0;
  }
  const double* wk = q.w + (m - nc);
  for (int j = threadIdx.x; j < nc; j += kNT)
    inverse_iteration(q.d, q.e, m, inverse_shift(wk, nc, j, tn), tn, nc, j, scr, Z);
  __syncthreads();
  // Gram-Schmidt against all earlier vectors: twice for an eigenvalue closer than 1e-3 of the
  // norm to its predecessor, once for the others.  Those are orthogonal to rounding over the
  // gap (1e-13), but left at that the overlap's 1e-13 reached some results: relative error of a
  // c8 a4 v61 n3 pass 1.1e-11 on one of six inputs, 2.8e-13 with the pass.  It costs 2 to 4 per
  // cent of the smallest solves.
  const double ctol = 1e-3 * tn;
  double* part = q.lo;                         // the brackets are no longer needed
  for (int c = 1; c < nc; ++c) {
    const int passes = wk[c] - wk[c - 1] > ctol ? 1 : 2;
    for (int pass = 0; pass < passes; ++pass) {
      for (int r0 = 0; r0 < c; r0 += 32) {
        const int r = r0 + lane;
        double a0 = 0.0, a1 = 0.0;
        if (r < c) {
          int i = warp;
          for (; i + kNW < m; i += 2 * kNW) {
            a0 = fma(Z[i * nc + r], Z[i * nc + c], a0);
            a1 = fma(Z[(i + kNW) * nc + r], Z[(i + kNW) * nc + c], a1);
          }
          if (i < m) a0 = fma(Z[i * nc + r], Z[i * nc + c], a0);
        }
        sh[8 + warp * 32 + lane] = a0 + a1;
        __syncthreads();
        if (warp == 0 && r < c) {
          double t = 0.0;
#pragma unroll
          for (int g = 0; g < kNW; ++g) t += sh[8 + g * 32 + lane];
          part[r] = t;
        }
        __syncthreads();
      }
      for (int i = threadIdx.x; i < m; i += kNT) {
        const double* zr = Z + i * nc;
        double a0 = 0.0, a1 = 0.0;
        int r = 0;
        for (; r + 1 < c; r += 2) {
          a0 = fma(part[r], zr[r], a0);
          a1 = fma(part[r + 1], zr[r + 1], a1);
        }
        if (r < c) a0 = fma(part[r], zr[r], a0);
        Z[i * nc + c] -= a0 + a1;
      }
      __syncthreads();
    }
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < m; i += 32) s = fma(Z[i * nc + c], Z[i * nc + c], s);
      s = warp_sum(s);
      const double f = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
      for (int i = lane; i < m; i += 32) Z[i * nc + c] *= f;
    }
    __syncthreads();
  }
  polish(m, nc, tn, wk, Z, scr, q);
  for (int j = threadIdx.x; j < m; j += kNT) q.w[j] *= unscale;
  __syncthreads();
  // back-transformation Z <- H_0 ... H_{m-3} Z: lanes over 32 columns, the block's warps
  // split over column chunks and row groups
  const int nch = (nc + 31) / 32;              // column chunks
  const int gr = max(1, kNW / nch);            // row groups a chunk
  for (int k = m - 3; k >= 0; --k) {
    const int n1 = m - k - 1;
    const double* u = A + k * ld + k + 1;
    const double t = q.tau[k];
    if (t == 0.0) continue;                    // the same for every thread
    for (int w0 = warp; w0 < nch * gr; w0 += kNW) {
      const int c = (w0 % nch) * 32 + lane, g = w0 / nch;
      double a0 = 0.0, a1 = 0.0;
      if (c < nc) {
        int i = g;
        for (; i + gr < n1; i += 2 * gr) {
          a0 = fma(u[i], Z[(k + 1 + i) * nc + c], a0);
          a1 = fma(u[i + gr], Z[(k + 1 + i + gr) * nc + c], a1);
        }
        if (i < n1) a0 = fma(u[i], Z[(k + 1 + i) * nc + c], a0);
      }
      sh[8 + w0 * 32 + lane] = a0 + a1;
    }
    __syncthreads();
    for (int w0 = warp; w0 < nch * gr; w0 += kNW) {
      const int c = (w0 % nch) * 32 + lane, g = w0 / nch;
      double r = 0.0;
      for (int h = 0; h < gr; ++h) r += sh[8 + (h * nch + w0 % nch) * 32 + lane];
      r *= t;
      if (c < nc)
        for (int i = g; i < n1; i += gr)
          Z[(k + 1 + i) * nc + c] = fma(-u[i], r, Z[(k + 1 + i) * nc + c]);
    }
    __syncthreads();
  }
  return nk;
}

// Shared memory of an m-row problem: A [m][m | 1], Z [m][m], the vectors.
__device__ __forceinline__ Vecs layout(double* sm, int m, double*& Z) {
  Z = sm + (long)m * (m | 1);
  double* v = Z + (long)m * m;
  Vecs q;
  q.d = v; q.e = v + m; q.e2 = v + 2 * m; q.tau = v + 3 * m; q.w = v + 4 * m;
  q.u = v + 5 * m; q.p = v + 6 * m; q.lo = v + 7 * m; q.hi = v + 8 * m;
  q.df = reinterpret_cast<float*>(v + 9 * m);
  q.ef = q.df + m;
  return q;
}

__global__ void __launch_bounds__(kNT)
k_sector_block(const SectorJob* __restrict__ jobs, int* __restrict__ info) {
  extern __shared__ double sm[];
  __shared__ double sh[8 + kNT];
  const SectorJob J = jobs[blockIdx.x];
  const int m = J.msec, ld = m | 1;
  double* A = sm;
  double* Z;
  const Vecs q = layout(sm, m, Z);
  const long mf = J.m, mm = mf * mf;
  auto element = [&](const double* in, int i, int j) {   // sym(in_id + sgn in_sw), selected rows
    const long ri = J.Lsel < 0 ? i : (long)i * J.n + J.Lsel;
    const long rj = J.Lsel < 0 ? j : (long)j * J.n + J.Lsel;
    const double x = in[ri * mf + rj] + J.sgn * in[mm + ri * mf + rj];
    const double y = in[rj * mf + ri] + J.sgn * in[mm + rj * mf + ri];
    return 0.5 * (x + y);
  };
  for (int t = threadIdx.x; t < m * m; t += kNT) A[(t / m) * ld + t % m] = element(J.S, t / m, t % m);
  __syncthreads();
  int nz;
  const int nk = eig_block(A, ld, m, J.thresh, Z, J.scr, q, sh, nz);
  if (nk <= 0) {
    if (threadIdx.x == 0) { info[2 * blockIdx.x] = 0; info[2 * blockIdx.x + 1] = nk; }
    return;
  }
  // X = Q s^(-1/2) in J.X and back in Z; F over A
  for (int t = threadIdx.x; t < nk; t += kNT) q.u[t] = 1.0 / sqrt(q.w[m - nk + t]);
  __syncthreads();
  for (int t = threadIdx.x; t < m * nk; t += kNT)
    J.X[t] = Z[(t / nk) * nz + nz - nk + t % nk] * q.u[t % nk];
  __syncthreads();
  for (int t = threadIdx.x; t < m * nk; t += kNT) Z[t] = J.X[t];
  for (int t = threadIdx.x; t < m * m; t += kNT) A[(t / m) * ld + t % m] = element(J.F, t / m, t % m);
  __syncthreads();
  block_mm(m, nk, m, A, ld, 1, Z, nk, 1, J.scr);                   // F X (through L2)
  __syncthreads();
  for (int t = threadIdx.x; t < m * nk; t += kNT) A[t] = J.scr[t];
  __syncthreads();
  double* Ft = J.scr + (long)m * m;
  block_mm(nk, nk, m, Z, 1, nk, A, nk, 1, Ft);                     // X^T F X
  __syncthreads();
  const int ld2 = nk | 1;
  for (int t = threadIdx.x; t < nk * nk; t += kNT) {
    const int i = t / nk, j = t % nk;
    A[i * ld2 + j] = 0.5 * (Ft[t] + Ft[j * nk + i]);
  }
  __syncthreads();
  const int nf = eig_block(A, ld2, nk, -1e300, Z, J.scr, q, sh, nz);
  if (nf != nk) {
    if (threadIdx.x == 0) { info[2 * blockIdx.x] = 0; info[2 * blockIdx.x + 1] = -1; }
    return;
  }
  for (int t = threadIdx.x; t < nk; t += kNT) J.omega[t] = q.w[t];
  block_mm(m, nk, nk, J.X, nk, 1, Z, nk, 1, J.Y);                  // Y = X P
  if (threadIdx.x == 0) { info[2 * blockIdx.x] = nk; info[2 * blockIdx.x + 1] = 0; }
}

// Eigenpairs of one matrix A [m][m]: w [m], V [m][nk] of the eigenvalues >= wmin; info = {nk,
// -1 on NaN}.  scr: 5 m^2 doubles.
__global__ void __launch_bounds__(kNT)
k_eig_block(const double* __restrict__ Ag, int m, double wmin, double* __restrict__ w,
            double* __restrict__ V, double* __restrict__ scr, int* __restrict__ info) {
  extern __shared__ double sm[];
  __shared__ double sh[8 + kNT];
  const int ld = m | 1;
  double* Z;
  const Vecs q = layout(sm, m, Z);
  for (int t = threadIdx.x; t < m * m; t += kNT)
    sm[(t / m) * ld + t % m] = 0.5 * (Ag[t] + Ag[(t % m) * m + t / m]);
  __syncthreads();
  int nz;
  const int nk = eig_block(sm, ld, m, wmin, Z, scr, q, sh, nz);
  if (threadIdx.x == 0) {
    info[0] = max(nk, 0);
    info[1] = nk < 0 ? -1 : 0;
  }
  if (nk < 0) return;
  for (int t = threadIdx.x; t < m; t += kNT) w[t] = q.w[t];
  for (int t = threadIdx.x; t < m * nk; t += kNT) V[t] = Z[(t / nk) * nz + nz - nk + t % nk];
}

size_t sector_smem(int m) {
  return sizeof(double) * ((size_t)m * (m | 1) + (size_t)m * m + (size_t)kNVec * m);
}

}  // namespace

size_t sector_block_scratch(int msec) { return (size_t)msec * msec * 5 + 64; }

cudaError_t sector_block_launch(const SectorJob* jobs, int njobs, int mmax, int* info,
                                cudaStream_t s) {
  if (njobs <= 0) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(k_sector_block,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sector_smem(kSectorBlockMax));
  if (e != cudaSuccess) return e;
  ++launch_counter();
  k_sector_block<<<njobs, kNT, sector_smem(mmax), s>>>(jobs, info);
  return cudaGetLastError();
}

int sym_eig_block(const double* A, int m, double* w, double* V, double* work, cudaStream_t s,
                  double wmin, int* nkept) {
  if (nkept) *nkept = 0;
  if (m <= 0) return CASPT2_OK;
  if (m > kSectorBlockMax) return CASPT2_EINVAL;
  CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_eig_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sector_smem(kSectorBlockMax)));
  int* info = reinterpret_cast<int*>(work + (size_t)5 * m * m + 32);
  ++launch_counter();
  k_eig_block<<<1, kNT, sector_smem(m), s>>>(A, m, wmin, w, V, work, info);
  CASPT2_CUDA_TRY(cudaGetLastError());
  int h[2] = {0, 0};
  CASPT2_CUDA_TRY(cudaMemcpyAsync(h, info, sizeof(h), cudaMemcpyDeviceToHost, s));
  CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
  if (h[1] != 0) return CASPT2_ENAN;
  if (nkept) *nkept = h[0];
  return CASPT2_OK;
}

}  // namespace caspt2
