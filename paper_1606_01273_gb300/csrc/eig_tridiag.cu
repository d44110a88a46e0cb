// FP64 symmetric eigensolver for the per-class overlap and Fock matrices
// (Sec. II.B: eigenvalues of the overlap below the threshold are truncated) above the size
// that one block solves (sector_block.cu):
//   1. Householder reduction to tridiagonal form, T = Q^T A Q (one reflector per step:
//      p = tau A22 v, w = p - (tau/2)(p.v) v, A22 -= v w^T + w v^T);
//   2. every eigenvalue of T from Sturm counts and minors (eig_dev.cuh, absolute accuracy
//      ~ eps ||T||);
//   3. eigenvectors of T by inverse iteration on the pivoted tridiagonal LU (one thread per
//      eigenvalue), Gram-Schmidt inside clusters of equal eigenvalues;
//   4. one Newton-Schulz step Z <- Z (3 - Z^T Z) / 2 to restore orthogonality to
//      rounding level (skipped when Z^T Z is already within 1e-13 of the identity);
//   5. back-transformation V = Q Z by applying the reflectors in reverse order.
#include <cstring>
#include <vector>

#include "class_ag.cuh"
#include "eig_dev.cuh"
#include "ozaki.cuh"
#include "linalg.cuh"

namespace caspt2 {

namespace {

constexpr int kT = 256;

int nblocks(long total, int threads = kT) {
  long b = (total + threads - 1) / threads;
  return (int)std::max<long>(1, std::min<long>(b, 152L * 32));
}

}  // namespace

// Grid-wide barrier for a cooperative launch, bounded: after kSpinLimit polls it sets
// *err and returns false so that every block can leave the kernel.
constexpr long kSpinLimit = 1L << 24;

__device__ bool grid_sync_bounded(unsigned* count, volatile unsigned* gen, int* err) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0) {
    unsigned g;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(g) : "l"(gen) : "memory");
    unsigned prev;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
                 : "=r"(prev) : "l"(count) : "memory");
    if (prev == gridDim.x - 1) {
      *count = 0;
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(gen), "r"(g + 1u) : "memory");
      ok = 1;
    } else {
      long it = 0;
      unsigned cur;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(gen) : "memory");
        if (cur != g) break;
        if (*(volatile int*)err != 0) break;
        if (++it > kSpinLimit) {
          atomicExch(err, 1);
          break;
        }
        if (it > 64) __nanosleep(32);
      }
      ok = (*(volatile int*)err == 0);
    }
  }
  __syncthreads();
  return ok != 0;
}

// Blocked Householder reduction, one cooperative launch per panel of b columns
// k0 .. k0+b-1 (the LAPACK dlatrd scheme, written from its definition): the trailing
// matrix is left as it stands during the panel and its true value is
// A22 - V W^T - W V^T, with V the panel's reflectors and W the vectors
// w = p - (tau/2)(p.v) v, p = tau (A22 - V W^T - W V^T) v.  After the panel the host
// applies A22 -= V W^T + W V^T as two FP64 GEMMs.  Per column k = k0 + j, three bounded
// grid barriers; blocks own contiguous runs of the rows (and of the columns of row k+1):
//   A: every block forms the reflector of row k from the row (already up to date) into
//      shared memory -- the reductions run in a fixed order, so every copy is the same;
//      block 0 stores it (vbuf row k, column j of Vr, tau, d, e);
//   B: p_raw = A22 v (a warp per half row, eight loads in flight per lane) and partial
//      sums of W^T v and V^T v;                                          | barrier
//   C: p = tau (p_raw - V (W^T v) - W (V^T v)) (a warp per owned row, lanes over the
//      panel columns) and partial sums of p.v;                           | barrier
//   D: alpha = (tau/2) p.v, W[:, j] = p - alpha v, and the owned columns of row k+1
//      brought up to date with the panel's columns 0..j.                 | barrier
// W and Vr are [m][nb] row-major (Vr holds the panel's reflectors by row, so that a row's
// panel entries are contiguous); p [m]; pr [2][m]; part [grid][2 nb + 1]; sync[0..1] barrier,
// [2] error.  Dynamic shared memory: v [m].
constexpr int kLatrdPanel = 64;
__global__ void __launch_bounds__(512, 2)
k_latrd(double* __restrict__ A, int m, int k0, int b, double* __restrict__ vbuf,
        double* __restrict__ tau, double* __restrict__ d, double* __restrict__ e,
        double* __restrict__ W, double* __restrict__ Vr, double* __restrict__ p,
        double* __restrict__ pr, double* __restrict__ part, unsigned* sync) {
  constexpr int nb = kLatrdPanel;
  extern __shared__ double vs[];                      // v of the current column, by row
  __shared__ double red[32];
  __shared__ double sh[4];
  __shared__ double xy[2 * nb];
  __shared__ double rk[2 * nb];                       // row k+1 of V and W (panel columns)
  int* err = reinterpret_cast<int*>(sync + 2);
  const int G = gridDim.x, bid = blockIdx.x;
  const int warp = (bid * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int nw = (G * blockDim.x) >> 5;
  const int wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  for (int j = 0; j < b; ++j) {
    const int k = k0 + j;
    const int n1 = m - k - 1;
    // ---- A: reflector of row k (every block; block 0 stores it)
    {
      const double* x = A + (long)k * m + k + 1;
      double s2 = 0.0;
      for (int i = 1 + threadIdx.x; i < n1; i += blockDim.x) {
        const double xi = __ldcg(x + i);
        s2 = fma(xi, xi, s2);
      }
      s2 = block_sum(s2, red);
      if (threadIdx.x == 0) {
        const double alpha = __ldcg(x);
        double beta, t, scale;
        if (s2 == 0.0) { beta = alpha; t = 0.0; scale = 0.0; }
        else {
          beta = -copysign(sqrt(alpha * alpha + s2), alpha);
          t = (beta - alpha) / beta;
          scale = 1.0 / (alpha - beta);
        }
        sh[0] = t;
        sh[1] = scale;
        if (bid == 0) {
          tau[k] = t;
          d[k] = __ldcg(A + (long)k * m + k);
          e[k] = beta;
        }
      }
      __syncthreads();
      const double scale = sh[1];
      for (int i = threadIdx.x; i < n1; i += blockDim.x) {
        const double vi = (i == 0) ? 1.0 : __ldcg(x + i) * scale;
        vs[k + 1 + i] = vi;
        if (bid == 0) {
          vbuf[(long)k * m + k + 1 + i] = vi;
          Vr[(long)(k + 1 + i) * nb + j] = vi;
        }
      }
      __syncthreads();
    }
    const double t = sh[0];
    const int R = (n1 + G - 1) / G;                   // rows (and row-k+1 columns) owned
    const int r0 = k + 1 + bid * R, r1 = min(m, r0 + R);
    // ---- B: p_raw = A22 v over rows >= k+1 as two half-row items per row (a warp per
    //      item, eight loads in flight per lane; pr holds the halves, [0, m) and [m, 2m));
    //      partials of W^T v, V^T v (columns l < j)
    {
      const int n1h = ((n1 + 1) / 2 + 31) / 32 * 32;
      for (int it = warp; it < 2 * n1; it += nw) {
        const int i = it >> 1, half = it & 1;
        const double* row = A + (long)(k + 1 + i) * m;
        const int qe = half ? m : min(m, k + 1 + n1h);
        double sa[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) sa[u] = 0.0;
        int q = k + 1 + (half ? n1h : 0) + lane;
        for (; q + 7 * 32 < qe; q += 8 * 32) {
          double av[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) av[u] = __ldcg(row + q + 32 * u);
#pragma unroll
          for (int u = 0; u < 8; ++u) sa[u] = fma(av[u], vs[q + 32 * u], sa[u]);
        }
        for (; q < qe; q += 32) sa[0] = fma(__ldcg(row + q), vs[q], sa[0]);
        double sum = ((sa[0] + sa[1]) + (sa[2] + sa[3])) + ((sa[4] + sa[5]) + (sa[6] + sa[7]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
        if (lane == 0) pr[half * m + k + 1 + i] = sum;
      }
    }
    if (threadIdx.x < 2 * j) {
      const int tq = threadIdx.x;
      const double* src = tq < j ? W + tq : Vr + (tq - j);
      double acc = 0.0;
      for (int i = r0; i < r1; ++i) acc = fma(__ldcg(src + (long)i * nb), vs[i], acc);
      part[(long)bid * (2 * nb + 1) + tq] = acc;
    }
    if (!grid_sync_bounded(sync, sync + 1, err)) return;
    // ---- C: p = tau (p_raw - V x - W y), x = W^T v, y = V^T v; partials of p . v
    //      (each x, y entry summed over the blocks' partials by one warp: lanes stride the
    //      blocks, then a fixed shuffle tree)
    for (int q = wib; q < 2 * j; q += wpb) {
      double acc = 0.0;
      for (int g = lane; g < G; g += 32) acc += __ldcg(part + (long)g * (2 * nb + 1) + q);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) xy[q] = acc;
    }
    __syncthreads();
    {
      double sp = 0.0;
      for (int i = r0 + wib; i < r1; i += wpb) {
        double c = 0.0;
        for (int l = lane; l < j; l += 32)
          c = fma(__ldcg(Vr + (long)i * nb + l), xy[l], fma(__ldcg(W + (long)i * nb + l), xy[j + l], c));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        const double pv = t * ((__ldcg(pr + i) + __ldcg(pr + m + i)) - c);
        if (lane == 0) p[i] = pv;
        sp = fma(pv, vs[i], sp);
      }
      sp = block_sum(lane == 0 ? sp : 0.0, red);
      if (threadIdx.x == 0) part[(long)bid * (2 * nb + 1) + 2 * nb] = sp;
    }
    if (!grid_sync_bounded(sync, sync + 1, err)) return;
    // ---- D: alpha = (tau/2) p.v (fixed order over the blocks), W[:, j] = p - alpha v;
    //         the owned columns of row k+1 brought up to date (not after the panel's last
    //         column: the trailing GEMM update takes over there)
    if (wib == 0) {
      double sum = 0.0;
      for (int g = lane; g < G; g += 32) sum += __ldcg(part + (long)g * (2 * nb + 1) + 2 * nb);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) sh[2] = 0.5 * t * sum;
    }
    __syncthreads();
    const double alpha = sh[2];
    for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x)
      W[(long)i * nb + j] = __ldcg(p + i) - alpha * vs[i];
    if (bid == 0)
      for (int i = threadIdx.x; i <= k; i += blockDim.x) W[(long)i * nb + j] = 0.0;
    if (j + 1 < b) {
      const int k1 = k + 1;
      // row k1 of V and W over l <= j (W[k1][j] formed here; p[k1] is visible)
      for (int l = threadIdx.x; l <= j; l += blockDim.x) {
        rk[l] = (l == j) ? vs[k1] : __ldcg(Vr + (long)k1 * nb + l);
        rk[nb + l] = (l == j) ? __ldcg(p + k1) - alpha * vs[k1] : __ldcg(W + (long)k1 * nb + l);
      }
      __syncthreads();
      for (int i = r0 + wib; i < r1; i += wpb) {
        double c = 0.0;
        for (int l = lane; l < j; l += 32)
          c = fma(rk[l], __ldcg(W + (long)i * nb + l), fma(rk[nb + l], __ldcg(Vr + (long)i * nb + l), c));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0) {
          const double wij = __ldcg(p + i) - alpha * vs[i];
          A[(long)k1 * m + i] = __ldcg(A + (long)k1 * m + i) - c - (rk[j] * wij + rk[nb + j] * vs[i]);
        }
      }
    }
    if (!grid_sync_bounded(sync, sync + 1, err)) return;
  }
}

// Householder reflector of x[0..n1) (x[0] = alpha): tau, beta and v (v[0] = 1) written
// by every calling block; the reduction order is fixed, so all blocks obtain bitwise
// identical results from identical x.
__device__ void house_vec(const double* __restrict__ x, int n1, double* __restrict__ v,
                          double* red, double* sh) {
  double s = 0.0;
  for (int i = 1 + threadIdx.x; i < n1; i += blockDim.x) s += x[i] * x[i];
  s = block_sum(s, red);
  if (threadIdx.x == 0) {
    const double alpha = x[0];
    double beta, t, scale;
    if (s == 0.0) { beta = alpha; t = 0.0; scale = 0.0; }
    else {
      beta = -copysign(sqrt(alpha * alpha + s), alpha);
      t = (beta - alpha) / beta;
      scale = 1.0 / (alpha - beta);
    }
    sh[0] = t;
    sh[1] = scale;
    sh[2] = beta;
  }
  __syncthreads();
  const double scale = sh[1];
  for (int i = threadIdx.x; i < n1; i += blockDim.x) v[i] = (i == 0) ? 1.0 : x[i] * scale;
  __syncthreads();
}

// Bounded barrier of all blocks of a cooperative launch: arrivals add to one counter that only
// grows, and every block polls it for G times the number of barriers passed (target).  One
// trip to L2 for the arrival and one for the poll, where a reset counter and a generation
// word take four.  A wait that gives up sets *err, which the others see in theirs.
__device__ bool grid_sync_count(unsigned* count, unsigned target, int* err) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    for (long it = 0;; ++it) {
      unsigned cur;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(count) : "memory");
      if (cur >= target) break;
      if ((it & 63) == 63 && *(volatile int*)err != 0) { ok = 0; break; }
      if (it > kSpinLimit) {
        atomicExch(err, 1);
        ok = 0;
        break;
      }
      if (it > 512) __nanosleep(32);
    }
  }
  __syncthreads();
  return ok != 0;
}

// Sum over the lanes of an aligned group of `width` (a power of two), in every lane.
__device__ __forceinline__ double group_sum(double v, int width) {
  for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Householder reduction with the matrix resident in shared memory: block b owns the
// rows r = b (mod gridDim.x).  One bounded grid barrier per step:
//   p_i = tau sum_j A_ij v_j for owned rows (published)                | barrier
//   every block: w = p - (tau/2)(p.v) v, and — redundantly — the update of row k+1
//   (published by its owner after the previous step) with the norm of its trailing part; the
//   next reflector's scalars by warp 0 while the other warps update the owned rows; the
//   owner of row k+2 publishes it.
// Shared layout: rows [nloc][m], v[m], w[m] (they change places each step), r[m] (all indexed
// by absolute column).  pbuf[2][m], rowbuf[2][m] are double-buffered by step parity; sync[0]
// barrier count, sync[2] error flag.
//
// What bounds it: at m = 1536 a third of the time is the FP64 unit (3 m^2 / 152 lane operations a
// block and step), the rest, and below m = 400 nearly all of it, the chain of a step: barrier,
// two block sums and the reflector's scalars.  An FP64 warp instruction takes 64 clocks of a
// sub-partition whether its lanes carry anything or not, so a block sum costs 5 x 64 clocks a
// warp and sub-partition: as few warps as the rows need (tridiag_threads).
__global__ void __launch_bounds__(512)
k_tridiag_smem(const double* __restrict__ A, int m, double* __restrict__ vbuf,
               double* __restrict__ tau, double* __restrict__ d, double* __restrict__ e,
               double* __restrict__ pbuf, double* __restrict__ rowbuf, unsigned* sync) {
  extern __shared__ double smem[];
  __shared__ double red[32], red2[32];
  __shared__ double sh[4];
  int* err = reinterpret_cast<int*>(sync + 2);
  const int G = gridDim.x, b = blockIdx.x;
  const int nloc = (m - b + G - 1) / G;            // rows b, b+G, ...
  double* rows = smem;
  double* v = rows + (long)((m + G - 1) / G) * m;
  double* w = v + m;                               // p of this step (all rows)
  double* r = w + m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  for (long q = threadIdx.x; q < (long)nloc * m; q += blockDim.x) {
    const int li = q / m, j = q % m;
    rows[q] = A[(long)(b + li * G) * m + j];
  }
  // reflector of row 0 (every block from the input)
  for (int j = threadIdx.x; j < m; j += blockDim.x) r[j] = A[j];
  __syncthreads();
  house_vec(r + 1, m - 1, v + 1, red, sh);
  double t = sh[0];
  if (b == 0) {
    for (int i = threadIdx.x; i < m - 1; i += blockDim.x) vbuf[1 + i] = v[1 + i];
    if (threadIdx.x == 0) { tau[0] = t; d[0] = r[0]; e[0] = sh[2]; }
  }
  unsigned target = 0;
  for (int k = 0; k + 2 < m; ++k) {
    const int k1 = k + 1, k2 = k + 2;
    // p = tau A v for the owned trailing rows (one warp per row, four partial sums)
    const int lfirst = (k1 - b + G - 1) / G;       // first owned row index >= k+1
    for (int li = lfirst + warp; li < nloc; li += nwarp) {
      const double* row = rows + (long)li * m;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      int j = k1 + lane;
      for (; j + 96 < m; j += 128) {
        s0 = fma(row[j], v[j], s0);
        s1 = fma(row[j + 32], v[j + 32], s1);
        s2 = fma(row[j + 64], v[j + 64], s2);
        s3 = fma(row[j + 96], v[j + 96], s3);
      }
      for (; j < m; j += 32) s0 = fma(row[j], v[j], s0);
      const double s = group_sum((s0 + s1) + (s2 + s3), 32);
      if (lane == 0) pbuf[(long)(k & 1) * m + b + li * G] = t * s;
    }
    target += (unsigned)G;
    if (!grid_sync_count(sync, target, err)) return;
    // g = (tau/2) p.v; with w = p - g v the update A -= v w^T + w v^T reads
    // A_ij -= v_i p_j + (p_i - 2 g v_i) v_j  (two FMAs per element); the old row k+1 (the
    // copy published before the barrier) comes in with p
    const double* old = (k == 0) ? A + (long)k1 * m : rowbuf + (long)(k1 & 1) * m;
    double s = 0.0;
#pragma unroll 4
    for (int j = k1 + threadIdx.x; j < m; j += blockDim.x) {
      const double pj = __ldcg(pbuf + (long)(k & 1) * m + j), oj = __ldcg(old + j);
      w[j] = pj;
      r[j] = oj;
      s = fma(pj, v[j], s);
    }
    s = group_sum(s, 32);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    const double g2 = t * group_sum(red[lane & (nwarp - 1)], nwarp);   // 2 g
    // row k+1 after this step and the square of its part right of the subdiagonal
    double q = 0.0;
    {
      const double vi = v[k1], bi = fma(-g2, vi, w[k1]);
#pragma unroll 4
      for (int j = k1 + threadIdx.x; j < m; j += blockDim.x) {
        const double x = fma(-bi, v[j], fma(-vi, w[j], r[j]));
        r[j] = x;
        if (j > k2) q = fma(x, x, q);
      }
    }
    const bool next = k + 3 < m;
    if (next) {
      q = group_sum(q, 32);
      if (lane == 0) red2[warp] = q;
    }
    __syncthreads();
    if (next && warp == 0) {
      // beta = -sign(alpha) |x|, tau = 1 + |alpha| / |x|, v = x / (alpha - beta) with v_0 = 1
      q = group_sum(red2[lane & (nwarp - 1)], nwarp);
      const double al = r[k2], sig = fma(al, al, q);
      double beta = al, tn = 0.0, scale = 0.0;
      if (q != 0.0 && !(sig < 1e-280)) {
        double nr, ir;
        root_and_recip(sig, nr, ir);
        beta = -copysign(nr, al);
        tn = fma(fabs(al), ir, 1.0);
        scale = copysign(recip(fabs(al) + nr), al);
      }
      if (lane == 0) { sh[0] = tn; sh[1] = scale; sh[2] = beta; }
    }
    // update of the owned rows
    for (int li = lfirst; li < nloc; ++li) {
      const int i = b + li * G;
      const double vi = v[i], bi = fma(-g2, vi, w[i]);
      double* row = rows + (long)li * m;
#pragma unroll 4
      for (int j = k1 + threadIdx.x; j < m; j += blockDim.x)
        row[j] = fma(-bi, v[j], fma(-vi, w[j], row[j]));
    }
    __syncthreads();
    // the owner of row k+2 publishes it for the next step
    if ((k2 % G) == b) {
      const double* row = rows + (long)(k2 / G) * m;
      for (int j = k2 + threadIdx.x; j < m; j += blockDim.x)
        rowbuf[(long)(k2 & 1) * m + j] = row[j];
    }
    if (next) {
      // next reflector from row k+1's trailing part, in the place of p
      t = sh[0];
      const double scale = sh[1];
      for (int j = k2 + threadIdx.x; j < m; j += blockDim.x) {
        const double x = j == k2 ? 1.0 : r[j] * scale;
        w[j] = x;
        if (b == 0) vbuf[(long)k1 * m + j] = x;
      }
      double* x = v;
      v = w;
      w = x;
      if (b == 0 && threadIdx.x == 0) { tau[k1] = t; d[k1] = r[k1]; e[k1] = sh[2]; }
    } else if (b == 0 && threadIdx.x == 0) {
      d[m - 2] = r[m - 2];
      e[m - 2] = r[m - 1];
    }
    __syncthreads();
  }
  // last diagonal element from its owner
  if (m >= 2 && ((m - 1) % G) == b && threadIdx.x == 0) {
    d[m - 1] = rows[(long)((m - 1) / G) * m + m - 1];
    e[m - 1] = 0.0;
  }
}

// Threads of a block of k_tridiag_smem: with up to three rows a block the block sums decide
// (m = 216: 1.01 ms with 128, 1.04 with 256, 1.29 with 512 threads; 1.58 before with 512; m = 384:
// 2.08, 2.09, 2.47), with more the rows (m = 864: 7.3, 6.3, 7.2 ms; m = 1536: 22.5, 17.7, 18.7 ms).
int tridiag_threads(int m, int G) { return (m + G - 1) / G <= 3 ? 128 : 256; }

// Shared memory of k_tridiag_smem for m columns on G blocks (0 if it does not fit).
constexpr size_t kTridiagSmemMax = 200ull * 1024;
constexpr size_t kBisectSmemMax = 200ull * 1024;    // d and e^2 of the tridiagonal matrix
constexpr size_t kBackSmemMax = 200ull * 1024;      // resident columns of the back-transform
size_t tridiag_smem_bytes(int m, int G) {
  const size_t b = 8ull * ((size_t)((m + G - 1) / G) * m + 3ull * m);
  return b <= kTridiagSmemMax ? b : 0;
}

__global__ void k_tail(const double* __restrict__ A, int m, double* d, double* e) {
  if (threadIdx.x != 0) return;
  if (m >= 2) {
    d[m - 2] = A[(long)(m - 2) * m + m - 2];
    e[m - 2] = A[(long)(m - 2) * m + m - 1];
  }
  d[m - 1] = A[(long)(m - 1) * m + m - 1];
  e[m - 1] = 0.0;
}

__global__ void k_e2(const double* __restrict__ e, int m, double* __restrict__ e2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) e2[i] = (i < m - 1) ? e[i] * e[i] : 0.0;
}

// Eigenvalues of T, eight lanes each: single-precision brackets, then FP64 (eig_dev.cuh).
// A warp's FP64 instruction occupies its sub-partition for 64 clocks, so the number of
// Sturm evaluations one after the other decides: 4 to 7 in place of the 12 passes of an FP64
// octasection.  Dynamic shared memory: d, e^2 and their float copies.
__global__ void k_eigenvalues(const double* __restrict__ dg, const double* __restrict__ e2g,
                              int m, double glo, double ghi, double tol, double wmin,
                              double* __restrict__ w) {
  extern __shared__ double sde[];
  float* sdf = reinterpret_cast<float*>(sde + 2 * m);
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    sde[i] = dg[i];
    sde[m + i] = e2g[i];
    sdf[i] = (float)dg[i];
    sdf[m + i] = (float)e2g[i];
  }
  __syncthreads();
  const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const int j = min(g, m - 1);
  float flo, fhi;
  bisect_f32(sdf, sdf + m, m, j, glo, ghi, flo, fhi);
  const double x = eigenvalue_f64_group(sde, sde + m, m, j, glo, ghi, flo, fhi, tol, wmin);
  if (g < m && (threadIdx.x & 7) == 0) w[g] = x;
}

// Inverse iteration for the nc eigenvalues w[0..nc) (thread j, eig_dev.cuh); scr as there.
__global__ void k_inviter(const double* __restrict__ dg, const double* __restrict__ eg,
                          const double* __restrict__ w, int m, int nc, double tnorm,
                          double* __restrict__ scr, double* __restrict__ Z) {
  extern __shared__ double sde[];      // d[m], e[m] staged per block
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    sde[i] = dg[i];
    sde[m + i] = eg[i];
  }
  __syncthreads();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nc)
    inverse_iteration(sde, sde + m, m, inverse_shift(w, nc, j, tnorm), tnorm, nc, j, scr, Z);
}

// Orthonormalise each cluster of close eigenvalues (w sorted): the block of the cluster's
// first index takes the cluster's columns, in shared memory when they fit (else in place
// in Z), and applies classical Gram-Schmidt twice per vector (each pass projects the
// vector on all earlier cluster vectors at once), then normalises it.  Z is m x nc.
__global__ void __launch_bounds__(256)
k_cluster_cgs2(const double* __restrict__ w, int m, int nc, double tol, int smem_bytes,
               double* __restrict__ Z) {
  extern __shared__ double cs[];
  __shared__ double part[8][33];
  __shared__ double red[32];
  __shared__ double sc;
  const int j0 = blockIdx.x;
  if (j0 > 0 && w[j0] - w[j0 - 1] <= tol) return;            // not a start
  if (j0 + 1 >= nc || w[j0 + 1] - w[j0] > tol) return;         // singleton
  int j1 = j0 + 1;
  while (j1 + 1 < nc && w[j1 + 1] - w[j1] <= tol) ++j1;
  const int c = j1 - j0 + 1;
  const bool in_smem = ((long)m * c + c) * 8 <= smem_bytes;
  double* Zb = in_smem ? cs : Z + j0;          // column q of the cluster: Zb[i * ld + q]
  const long ld = in_smem ? c : nc;
  double* pk = in_smem ? cs + (long)m * c : cs;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (in_smem) {
    for (long t = threadIdx.x; t < (long)m * c; t += blockDim.x)
      cs[t] = Z[(t / c) * nc + j0 + t % c];
    __syncthreads();
  }
  for (int q = 0; q < c; ++q) {
    for (int pass = 0; pass < 2 && q > 0; ++pass) {
      // pk[r] = sum_i Zb[i][r] Zb[i][q] for r < q: lanes over 32 columns, warps over rows
      // (four independent partial sums each), fixed-order sums over the warps
      for (int r0 = 0; r0 < q; r0 += 32) {
        const int r = r0 + lane;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        if (r < q) {
          int i = wp;
          for (; i + 24 < m; i += 32) {
            a0 += Zb[i * ld + r] * Zb[i * ld + q];
            a1 += Zb[(i + 8) * ld + r] * Zb[(i + 8) * ld + q];
            a2 += Zb[(i + 16) * ld + r] * Zb[(i + 16) * ld + q];
            a3 += Zb[(i + 24) * ld + r] * Zb[(i + 24) * ld + q];
          }
          for (; i < m; i += 8) a0 += Zb[i * ld + r] * Zb[i * ld + q];
        }
        part[wp][lane] = (a0 + a1) + (a2 + a3);
        __syncthreads();
        if (wp == 0 && r < q) {
          double t = 0.0;
#pragma unroll
          for (int g = 0; g < 8; ++g) t += part[g][lane];
          pk[r] = t;
        }
        __syncthreads();
      }
      // Zb[i][q] -= sum_r pk[r] Zb[i][r]: one thread per row
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const double* zr = Zb + i * ld;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int r = 0;
        for (; r + 3 < q; r += 4) {
          a0 += pk[r] * zr[r];
          a1 += pk[r + 1] * zr[r + 1];
          a2 += pk[r + 2] * zr[r + 2];
          a3 += pk[r + 3] * zr[r + 3];
        }
        for (; r < q; ++r) a0 += pk[r] * zr[r];
        Zb[i * ld + q] -= (a0 + a1) + (a2 + a3);
      }
      __syncthreads();
    }
    double s2 = 0.0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) s2 += Zb[i * ld + q] * Zb[i * ld + q];
    s2 = block_sum(s2, red);
    if (threadIdx.x == 0) sc = (s2 > 0.0) ? 1.0 / sqrt(s2) : 0.0;
    __syncthreads();
    const double nr = sc;
    for (int i = threadIdx.x; i < m; i += blockDim.x) Zb[i * ld + q] *= nr;
    __syncthreads();
  }
  if (in_smem)
    for (long t = threadIdx.x; t < (long)m * c; t += blockDim.x)
      Z[(t / c) * nc + j0 + t % c] = cs[t];
}

// G[i][i] -= x
__global__ void k_sub_diag(double* __restrict__ G, int m, double x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) G[(long)i * m + i] -= x;
}

// G = 1.5 I - 0.5 G (in place)
// and dev = max |G - I| (order-independent integer maximum of the bit patterns)
__global__ void k_ns_coef(double* __restrict__ G, int m, unsigned long long* __restrict__ dev) {
  const long total = (long)m * m;
  unsigned long long mx = 0;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
       t += (long)gridDim.x * blockDim.x) {
    const bool diag = t / m == t % m;
    const double g = G[t];
    const unsigned long long b =
        (unsigned long long)__double_as_longlong(g - (diag ? 1.0 : 0.0)) & 0x7FFFFFFFFFFFFFFFull;
    mx = b > mx ? b : mx;
    G[t] = (diag ? 1.5 : 0.0) - 0.5 * g;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = y > mx ? y : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(dev, mx);
}

// Orthonormality probe of the eigenvector matrix Z (columns): with two fixed +-1 vectors
// r1, r2, dev = max_k |(Z^T Z r)_k - r_k| over both (two passes over Z instead of the m^3
// Gram product).  A column set orthonormal to within e gives dev <~ e sqrt(m); a larger
// dev sends the caller to the full Gram matrix.
__device__ __forceinline__ double probe_sign(int k, int which) {
  const unsigned h = (unsigned)k * 2654435761u + (which ? 0x9E3779B9u : 0x7F4A7C15u);
  return ((h >> 13) & 1u) ? 1.0 : -1.0;
}
// u[q][i] = sum_k Z[i][k] r_q[k]: a warp per row
__global__ void __launch_bounds__(256)
k_ortho_probe1(const double* __restrict__ Z, int m, int nc, double* __restrict__ u) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int i = warp; i < m; i += nw) {
    const double* row = Z + (long)i * nc;
    double s1 = 0.0, s2 = 0.0;
    for (int k = lane; k < nc; k += 32) {
      const double z = row[k];
      s1 = fma(z, probe_sign(k, 0), s1);
      s2 = fma(z, probe_sign(k, 1), s2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_down_sync(0xffffffffu, s1, o);
      s2 += __shfl_down_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) {
      u[i] = s1;
      u[m + i] = s2;
    }
  }
}
// w_q[c] = sum_i Z[i][c] u_q[i] (32 columns x 8 row groups per block, fixed-order sum over
// the groups) and dev = max |w_q[c] - r_q[c]| (integer maximum of the bit patterns)
__global__ void __launch_bounds__(256)
k_ortho_probe2(const double* __restrict__ Z, int m, int nc, const double* __restrict__ u,
               unsigned long long* __restrict__ dev) {
  __shared__ double part[2][8][33];
  const int cx = threadIdx.x & 31, rg = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + cx;
  double s1 = 0.0, s2 = 0.0;
  if (c < nc)
    for (int i = rg; i < m; i += 8) {
      const double z = Z[(long)i * nc + c];
      s1 = fma(z, u[i], s1);
      s2 = fma(z, u[m + i], s2);
    }
  part[0][rg][cx] = s1;
  part[1][rg][cx] = s2;
  __syncthreads();
  if (rg == 0 && c < nc) {
    double w1 = 0.0, w2 = 0.0;
    for (int g = 0; g < 8; ++g) {
      w1 += part[0][g][cx];
      w2 += part[1][g][cx];
    }
    const double e = fmax(fabs(w1 - probe_sign(c, 0)), fabs(w2 - probe_sign(c, 1)));
    const unsigned long long b = (unsigned long long)__double_as_longlong(e);
    if (e == e) atomicMax(dev, b);
    else atomicMax(dev, 0x7FF8000000000000ull);
  }
}

// Back-transformation V = H_0 ... H_{m-3} Z with each block owning cb consecutive columns of Z,
// resident in shared memory (column-major, zs[c][i]) for the whole reflector loop, and one warp
// per column: the warp forms v . z_c with a shuffle reduction and updates its column, so the block synchronises
// once per reflector, when the next reflector (double-buffered in shared memory by
// 8-byte cp.async copies) has landed.  Z is read and written once.
__global__ void __launch_bounds__(512)
k_backtransform_smem(const double* __restrict__ vbuf, const double* __restrict__ tau, int m,
                     int nc, int cb, double* __restrict__ Z) {
  extern __shared__ double zs[];                 // zs[cb][m], then vs[2][m]
  double* vs = zs + (long)cb * m;
  const int c0 = blockIdx.x * cb;
  const int ncol = min(cb, nc - c0);
  const int lane = threadIdx.x & 31, wc = threadIdx.x >> 5;
  const int nth = blockDim.x;
  for (long q = threadIdx.x; q < (long)m * cb; q += nth) {
    const int i = q / cb, c = q % cb;            // row-major walk of Z (coalesced per row)
    zs[(long)c * m + i] = c < ncol ? Z[(long)i * nc + c0 + c] : 0.0;
  }
  auto prefetch = [&](int k) {                   // v_k -> vs[k & 1]
    const int n1 = m - k - 1;
    const double* v = vbuf + (long)k * m + k + 1;
    double* dst = vs + (long)(k & 1) * m;
    for (int i = threadIdx.x; i < n1; i += nth) {
      const unsigned sa = (unsigned)__cvta_generic_to_shared(dst + i);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(v + i) : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  if (m >= 3) prefetch(m - 3);
  const bool act = wc < ncol;
  double* zc = zs + (long)wc * m;
  for (int k = m - 3; k >= 0; --k) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();                             // v_k visible; step k+1 done with vs[(k+1)&1]
    if (k > 0) prefetch(k - 1);
    if (!act) continue;
    const int n1 = m - k - 1;
    const double* v = vs + (long)(k & 1) * m;
    double* z = zc + k + 1;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int i = lane;
    for (; i + 96 < n1; i += 128) {
      s0 += v[i] * z[i];
      s1 += v[i + 32] * z[i + 32];
      s2 += v[i + 64] * z[i + 64];
      s3 += v[i + 96] * z[i + 96];
    }
    for (; i < n1; i += 32) s0 += v[i] * z[i];
    double sum = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const double r = sum * tau[k];
    for (int i2 = lane; i2 < n1; i2 += 32) z[i2] -= v[i2] * r;
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  for (long q = threadIdx.x; q < (long)m * cb; q += nth) {
    const int i = q / cb, c = q % cb;
    if (c < ncol) Z[(long)i * nc + c0 + c] = zs[(long)c * m + i];
  }
}

// Compact WY form of the panels of reflectors (Schreiber and Van Loan): H_k0 ... H_k0+b-1 =
// I - Vp T Vp^T with T upper triangular, T_ii = tau_i and
// T_{j,i} = -tau_i sum_{l = j..i-1} T_{j,l} (v_l . v_i) (j < i).  One block per panel of nb
// reflectors (the last one shorter), all panels at once; G[panel][l][i] = v_l . v_i is
// overwritten by T.  Column i of G is needed at step i only, so T takes its place in shared
// memory; eight lanes a row.  (One block of b threads a panel, each with a serial sum over
// global memory, took 0.51 ms a panel, one panel after the other.)
constexpr int kWyPanel = 128;       // reflectors per compact-WY panel
__global__ void __launch_bounds__(256)
k_wy_T(double* __restrict__ G, const double* __restrict__ tau, int nref) {
  extern __shared__ double t[];
  constexpr int nb = kWyPanel, ld = nb + 1;
  const int k0 = blockIdx.x * nb, b = min(nb, nref - k0);
  double* Gp = G + (long)blockIdx.x * nb * nb;
  for (int q = threadIdx.x; q < b * b; q += blockDim.x) t[(q / b) * ld + q % b] = Gp[(q / b) * nb + q % b];
  __syncthreads();
  const int sub = threadIdx.x & 7;
  for (int i = 0; i < b; ++i) {
    const double ti = tau[k0 + i];
    double res[nb / 32];
#pragma unroll
    for (int r = 0; r < nb / 32; ++r) {
      const int j = r * 32 + (threadIdx.x >> 3);
      double s0 = 0.0, s1 = 0.0;
      if (j < i) {
        int l = j + sub;
        for (; l + 8 < i; l += 16) {
          s0 = fma(t[j * ld + l], t[l * ld + i], s0);
          s1 = fma(t[j * ld + l + 8], t[(l + 8) * ld + i], s1);
        }
        if (l < i) s0 = fma(t[j * ld + l], t[l * ld + i], s0);
      }
      res[r] = 0.0;
      if (r * 32 + (threadIdx.x >> 5) * 4 < i) {        // whole warps
        double s = s0 + s1;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        res[r] = -ti * s;
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < nb / 32; ++r) {
      const int j = r * 32 + (threadIdx.x >> 3);
      if (sub == 0 && j < b) t[j * ld + i] = j < i ? res[r] : (j == i ? ti : 0.0);
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < b * b; q += blockDim.x) Gp[(q / b) * nb + q % b] = t[(q / b) * ld + q % b];
}

size_t sym_eig_tridiag_work(int m) { return (size_t)m * m * 9 + (size_t)m * 8 + 64; }

namespace {
constexpr int kWyMinSize = 1024;    // blocked back-transformation from this size up

// V <- H_0 H_1 ... H_{m-3} V as panels P_j = I - Vp T Vp^T applied last panel first:
// W = Vp^T V (rows below the panel start), W <- T W, V -= Vp W, three FP64 GEMMs per
// panel.  vbuf rows hold the reflectors with zeros left of their first entry, so a panel's
// rows of vbuf are Vp^T as it stands.  scratch >= 2 b nc + b (m + b) doubles.
int backtransform_wy(const double* vbuf, const double* tau, int m, int nc, double* V,
                     double* scratch, long scratch_size, cudaStream_t s, OzWork* oz) {
  const int nref = m - 2;
  const int nb = kWyPanel;
  const int npanel = (nref + nb - 1) / nb;
  double* W = scratch;
  double* W2 = W + (long)nb * nc;
  double* T = W2 + (long)nb * nc;                        // [panel][nb][nb]
  if ((T - scratch) + (long)npanel * nb * nb > scratch_size) return CASPT2_EINVAL;
  // every panel's T at once: Gram matrices (the last, shorter panel apart), then k_wy_T
  const int full = nref / nb, last = nref - full * nb;
  CASPT2_CUDA_TRY(dgemm(nb, nb, m, 1.0, vbuf, m, false, vbuf, m, true, 0.0, T, nb, s, full,
                        (long)nb * m, (long)nb * m, (long)nb * nb));
  if (last > 0) {
    const double* vl = vbuf + (long)full * nb * m;
    CASPT2_CUDA_TRY(dgemm(last, last, m, 1.0, vl, m, false, vl, m, true, 0.0,
                          T + (long)full * nb * nb, nb, s));
  }
  constexpr size_t tsm = sizeof(double) * kWyPanel * (kWyPanel + 1);
  CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_wy_T, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)tsm));
  ++launch_counter();
  k_wy_T<<<npanel, 256, tsm, s>>>(T, tau, nref);
  CASPT2_CUDA_TRY(cudaGetLastError());
  for (int k0 = ((nref - 1) / nb) * nb; k0 >= 0; k0 -= nb) {
    const int b = std::min(nb, nref - k0);
    const int r = m - k0 - 1;                            // rows k0+1 .. m-1
    const double* Vt = vbuf + (long)k0 * m;              // b x m, zeros left of each v
    const double* Tp = T + (long)(k0 / nb) * nb * nb;
    if (oz && oz->on) {
      // precision form: the two large products as FP64-accurate split products (the
      // eigenvalues are fixed before this step; only the vectors pass through it)
      const OzView va{Vt + k0 + 1, m, 1, r, 0};                  // rows l, K = row i
      const OzView vb{V + (long)(k0 + 1) * nc, 1, nc, r, 0};     // rows col, K = row i
      CASPT2_CUDA_TRY(oz_matmul(*oz, va, vb, false, b, nc, r, 1.0, 0.0, W, nc, s));
      CASPT2_CUDA_TRY(dgemm(b, nc, b, 1.0, Tp, nb, false, W, nc, false, 0.0, W2, nc, s));
      const OzView vp{Vt + k0 + 1, 1, m, b, 0};                  // rows i, K = l
      const OzView vw{W2, 1, nc, b, 0};                          // rows col, K = l
      CASPT2_CUDA_TRY(oz_matmul(*oz, vp, vw, false, r, nc, b, -1.0, 1.0, V + (long)(k0 + 1) * nc,
                                nc, s));
    } else {
      CASPT2_CUDA_TRY(dgemm(b, nc, r, 1.0, Vt + k0 + 1, m, false, V + (long)(k0 + 1) * nc, nc,
                            false, 0.0, W, nc, s));
      CASPT2_CUDA_TRY(dgemm(b, nc, b, 1.0, Tp, nb, false, W, nc, false, 0.0, W2, nc, s));
      CASPT2_CUDA_TRY(dgemm(r, nc, b, -1.0, Vt + k0 + 1, m, true, W2, nc, false, 1.0,
                            V + (long)(k0 + 1) * nc, nc, s));
    }
  }
  return CASPT2_OK;
}
}  // namespace

int sym_eig_tridiag(double* A, int m, double* w, double* V, double* work, cudaStream_t s,
                    KernelTimer* tm, OzWork* oz, double wmin, int* nkept) {
  if (nkept) *nkept = 0;
  if (m <= 0) return CASPT2_OK;
  const long mm = (long)m * m;
  double* vbuf = work;            // m*m reflectors
  double* Z = vbuf + mm;          // m*m eigenvectors of T
  double* G = Z + mm;             // m*m Gram / scratch
  double* u0 = G + mm;            // 5*m*m inverse-iteration scratch
  double* u1 = u0 + mm;
  double* u2 = u1 + mm;
  double* d = u2 + 3 * mm;
  double* e = d + m;
  double* e2 = e + m;
  double* tau = e2 + m;
  double* p = tau + m;
  double* r = p + m;
  // reflector rows are read whole by the blocked back-transformation: zero them first
  if (m >= kWyMinSize) CASPT2_CUDA_TRY(cudaMemsetAsync(vbuf, 0, sizeof(double) * mm, s));
  // 1. tridiagonalise (one cooperative launch for large matrices: rows resident in
  //    shared memory when they fit, else streamed through L2)
  int dev = 0, nsm = 0;
  CASPT2_CUDA_TRY(cudaGetDevice(&dev));
  CASPT2_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const int Gs = std::max(1, std::min(nsm, m));
  const size_t smem_b = tridiag_smem_bytes(m, Gs);
  if (smem_b > 0) {
    unsigned* sync = reinterpret_cast<unsigned*>(r);   // r is free until the back-transform
    double* pbuf = u0;                                 // u0.. are free until inverse iteration
    double* rowbuf = u0 + 2 * (long)m;
    // the attribute is global to the kernel: set the fixed maximum (never a per-launch
    // size) so that concurrent solves of different sizes cannot lower it under each other
    CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_tridiag_smem,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTridiagSmemMax));
    CASPT2_CUDA_TRY(cudaMemsetAsync(sync, 0, 4 * sizeof(unsigned), s));
    const double* Ac = A;
    void* args[] = {&Ac, (void*)&m, &vbuf, &tau, &d, &e, &pbuf, &rowbuf, &sync};
    ++launch_counter();
    if (tm && tm->e0) CASPT2_CUDA_TRY(cudaEventRecord(tm->e0, s));
    CASPT2_CUDA_TRY(cudaLaunchCooperativeKernel((void*)k_tridiag_smem, Gs,
                                                tridiag_threads(m, Gs), args, smem_b, s));
    if (tm && tm->e1) CASPT2_CUDA_TRY(cudaEventRecord(tm->e1, s));
    int herr = 0;
    CASPT2_CUDA_TRY(cudaMemcpyAsync(&herr, sync + 2, sizeof(int), cudaMemcpyDeviceToHost, s));
    CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
    if (herr != 0) return CASPT2_ETIMEOUT;
    if (tm && tm->e0) {
      float ms = 0.f;
      CASPT2_CUDA_TRY(cudaEventElapsedTime(&ms, tm->e0, tm->e1));
      tm->ms += ms;
      tm->flops += 4.0 / 3.0 * (double)m * m * m;   // Householder tridiagonalisation
      // the matrix read once and the reflectors (lower triangle) written once
      tm->bytes += 8.0 * m * m + 4.0 * m * (m - 1.0);
      ++tm->launches;
    }
  } else {
    // blocked reduction: panels of kLatrdPanel columns (one cooperative launch each) and
    // the trailing update as two FP64 GEMMs per panel
    unsigned* sync = reinterpret_cast<unsigned*>(r);   // r is free until the back-transform
    double* Wp = u0;                                   // [m][kLatrdPanel]
    double* pp = u1;
    double* pr = u1 + m;                               // [2][m] (the two row halves)
    double* part = u1 + 3 * (long)m;                   // [grid][2 panel + 1]
    double* Vr = u2;                                   // [m][kLatrdPanel]
    if (sizeof(double) * (size_t)m > kBisectSmemMax) return CASPT2_EINVAL;
    CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_latrd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kBisectSmemMax));
    int per = 0;
    CASPT2_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_latrd, 512,
                                                                  sizeof(double) * (size_t)m));
    // two blocks per SM when they fit (more warps in flight for the latency-bound
    // matrix-vector products), one otherwise
    const int grid = std::max(1, nsm * std::max(1, std::min(per, 2)));
    if ((long)grid * (2 * kLatrdPanel + 1) > mm - 3 * (long)m) return CASPT2_EINVAL;
    CASPT2_CUDA_TRY(cudaMemsetAsync(sync, 0, 4 * sizeof(unsigned), s));
    const int npanel = (m - 2 + kLatrdPanel - 1) / kLatrdPanel;
    if (tm && tm->e0) {
      while ((int)tm->pev.size() < 2 * npanel) {
        cudaEvent_t ev = nullptr;
        CASPT2_CUDA_TRY(cudaEventCreate(&ev));
        tm->pev.push_back(ev);
      }
      CASPT2_CUDA_TRY(cudaEventRecord(tm->e0, s));
    }
    std::vector<double> pbytes;
    for (int k0 = 0; k0 < m - 2; k0 += kLatrdPanel) {
      const int b = std::min(kLatrdPanel, m - 2 - k0);
      void* args[] = {&A, (void*)&m, (void*)&k0, (void*)&b, &vbuf, &tau, &d, &e, &Wp, &Vr, &pp,
                      &pr, &part, &sync};
      const int pi = k0 / kLatrdPanel;
      if (tm && tm->e0) {
        CASPT2_CUDA_TRY(cudaEventRecord(tm->pev[2 * pi], s));
        double by = 0.0;
        for (int j = 0; j < b; ++j) {
          const double n1 = (double)(m - k0 - j - 1);
          by += 8.0 * n1 * n1;
        }
        pbytes.push_back(by);
      }
      ++launch_counter();
      CASPT2_CUDA_TRY(cudaLaunchCooperativeKernel((void*)k_latrd, grid, 512, args,
                                                  sizeof(double) * (size_t)m, s));
      if (tm && tm->e0) CASPT2_CUDA_TRY(cudaEventRecord(tm->pev[2 * pi + 1], s));
      const int rr = m - k0 - b;
      if (rr > 0) {
        double* A22 = A + (long)(k0 + b) * m + k0 + b;
        const double* Vp = vbuf + (long)k0 * m + k0 + b;
        const double* Wr = Wp + (long)(k0 + b) * kLatrdPanel;
        CASPT2_CUDA_TRY(dgemm(rr, rr, b, -1.0, Vp, m, true, Wr, kLatrdPanel, true, 1.0, A22, m, s));
        CASPT2_CUDA_TRY(dgemm(rr, rr, b, -1.0, Wr, kLatrdPanel, false, Vp, m, false, 1.0, A22, m,
                              s));
      }
    }
    if (tm && tm->e1) CASPT2_CUDA_TRY(cudaEventRecord(tm->e1, s));
    int herr = 0;
    CASPT2_CUDA_TRY(cudaMemcpyAsync(&herr, sync + 2, sizeof(int), cudaMemcpyDeviceToHost, s));
    CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
    if (herr != 0) return CASPT2_ETIMEOUT;
    if (tm && tm->e0) {
      float ms = 0.f;
      CASPT2_CUDA_TRY(cudaEventElapsedTime(&ms, tm->e0, tm->e1));
      tm->ms += ms;
      tm->flops += 4.0 / 3.0 * (double)m * m * m;   // Householder tridiagonalisation
      tm->bytes += 8.0 * m * m + 4.0 * m * (m - 1.0);
      for (size_t q = 0; q < pbytes.size(); ++q) {
        float pm = 0.f;
        CASPT2_CUDA_TRY(cudaEventElapsedTime(&pm, tm->pev[2 * q], tm->pev[2 * q + 1]));
        tm->pms += pm;
        tm->pbytes += pbytes[q];
        ++tm->plaunches;
      }
      ++tm->launches;
    }
  }
  if (smem_b == 0) {
    ++launch_counter();
    k_tail<<<1, 32, 0, s>>>(A, m, d, e);
  }
  CASPT2_CUDA_TRY(cudaGetLastError());
  // Gershgorin interval and pivmin on the host (small vectors)
  std::vector<double> hd(m), he(m);
  CASPT2_CUDA_TRY(cudaMemcpyAsync(hd.data(), d, sizeof(double) * m, cudaMemcpyDeviceToHost, s));
  CASPT2_CUDA_TRY(cudaMemcpyAsync(he.data(), e, sizeof(double) * m, cudaMemcpyDeviceToHost, s));
  CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
  double glo = 1e300, ghi = -1e300, tnorm = 0.0;
  for (int i = 0; i < m; ++i) {
    const double r0 = (i > 0 ? fabs(he[i - 1]) : 0.0) + (i < m - 1 ? fabs(he[i]) : 0.0);
    glo = std::min(glo, hd[i] - r0);
    ghi = std::max(ghi, hd[i] + r0);
    tnorm = std::max(tnorm, fabs(hd[i]) + r0);
    if (!(hd[i] == hd[i]) || !(he[i] == he[i])) return CASPT2_ENAN;
  }
  const double pad = 2.2e-16 * std::max(1.0, tnorm) * 4.0 + 1e-300;
  glo -= pad;
  ghi += pad;
  // 2. eigenvalues
  ++launch_counter();
  k_e2<<<(m + 255) / 256, 256, 0, s>>>(e, m, e2);
  ++launch_counter();
  if (3 * sizeof(double) * (size_t)m > kBisectSmemMax) return CASPT2_EINVAL;
  CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_eigenvalues, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kBisectSmemMax));
  // blocks sized so that one wave covers all 8m lanes (the staged copy of the tridiagonal
  // matrix limits residency to one block per SM at the largest sizes)
  const int ev_t = (int)std::min<long>(1024, std::max<long>(32, ((8L * m + nsm - 1) / nsm + 31) / 32 * 32));
  k_eigenvalues<<<(unsigned)((8L * m + ev_t - 1) / ev_t), ev_t, 3 * sizeof(double) * m, s>>>(
      d, e2, m, glo, ghi, kEigTol * std::max(1.0, tnorm), nkept ? eig_guard(wmin, tnorm) : -1e300, w);
  CASPT2_CUDA_TRY(cudaGetLastError());
  // the vectors to return: all, or those of the eigenvalues at or above wmin (the last nk of
  // the ascending list); nc >= nk are formed (eig_guard)
  int j0 = 0, nk = m;
  if (nkept) {
    CASPT2_CUDA_TRY(cudaMemcpyAsync(hd.data(), w, sizeof(double) * m, cudaMemcpyDeviceToHost, s));
    CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
    while (j0 < m && hd[j0] < wmin) ++j0;
    *nkept = nk = m - j0;
    if (nk == 0) return CASPT2_OK;
    while (j0 > 0 && hd[j0 - 1] >= eig_guard(wmin, tnorm)) --j0;
  }
  const int nc = m - j0;
  const double* wk = w + j0;
  // 3. eigenvectors of T
  ++launch_counter();
  // one warp per block so that the m independent LU chains spread over the SMs
  CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_inviter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kBisectSmemMax));
  k_inviter<<<(nc + 31) / 32, 32, 2 * sizeof(double) * m, s>>>(d, e, wk, m, nc, tnorm, u0, Z);
  ++launch_counter();
  CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_cluster_cgs2, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kBisectSmemMax));
  {
    const int cbytes = (int)std::min<size_t>(kBisectSmemMax, 8ull * ((size_t)m * nc + nc));
    k_cluster_cgs2<<<nc, 256, cbytes, s>>>(wk, m, nc, 1e-12 * std::max(1.0, tnorm), cbytes, Z);
  }
  CASPT2_CUDA_TRY(cudaGetLastError());
  // 4. Newton-Schulz: Z <- Z (1.5 I - 0.5 Z^T Z), skipped when Z is already orthonormal to
  //    1e-13 (the step would change it by less than that)
  //    The probe Z^T Z r (two passes over Z) decides first; only when it is above 1e-13 is
  //    the m^3 Gram matrix formed and the element-wise test applied.
  unsigned long long* ns_dev = reinterpret_cast<unsigned long long*>(r + m);
  CASPT2_CUDA_TRY(cudaMemsetAsync(ns_dev, 0, sizeof(unsigned long long), s));
  ++launch_counter();
  k_ortho_probe1<<<nblocks(32L * m), kT, 0, s>>>(Z, m, nc, G);
  ++launch_counter();
  k_ortho_probe2<<<(nc + 31) / 32, 256, 0, s>>>(Z, m, nc, G, ns_dev);
  CASPT2_CUDA_TRY(cudaGetLastError());
  unsigned long long hdev = 0;
  CASPT2_CUDA_TRY(cudaMemcpyAsync(&hdev, ns_dev, sizeof(hdev), cudaMemcpyDeviceToHost, s));
  CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
  double dev_probe;
  std::memcpy(&dev_probe, &hdev, sizeof(double));
  if (!(dev_probe == dev_probe)) return CASPT2_ENAN;
  // V = the last nk columns of Z
  auto take_columns = [&]() {
    return cudaMemcpy2DAsync(V, sizeof(double) * nk, Z + (nc - nk), sizeof(double) * nc,
                             sizeof(double) * nk, m, cudaMemcpyDeviceToDevice, s);
  };
  if (dev_probe <= 1e-13) {
    CASPT2_CUDA_TRY(take_columns());
  } else {
    CASPT2_CUDA_TRY(cudaMemsetAsync(ns_dev, 0, sizeof(unsigned long long), s));
    CASPT2_CUDA_TRY(dgemm_sym(nc, m, 1.0, Z, nc, true, Z, nc, false, 0.0, G, nc, s));
    ++launch_counter();
    k_ns_coef<<<nblocks((long)nc * nc), kT, 0, s>>>(G, nc, ns_dev);
    CASPT2_CUDA_TRY(cudaGetLastError());
    CASPT2_CUDA_TRY(cudaMemcpyAsync(&hdev, ns_dev, sizeof(hdev), cudaMemcpyDeviceToHost, s));
    CASPT2_CUDA_TRY(cudaStreamSynchronize(s));
    double dev_ortho;
    std::memcpy(&dev_ortho, &hdev, sizeof(double));
    if (!(dev_ortho == dev_ortho)) return CASPT2_ENAN;
    if (dev_ortho <= 1e-13) {
      CASPT2_CUDA_TRY(take_columns());
    } else if (oz && oz->on) {
      // V = Z + Z Ec, Ec = (1/2)(I - Z^T Z) (G - I): the correction is of the size of the
      // orthogonality error, so a split product with S slices (error below about
      // 2^(1-7S) m max|Z| max|Ec|) is kept under 1e-17 with S = ceil((57 + log2(m dev/2)) / 7)
      ++launch_counter();
      k_sub_diag<<<(nc + 255) / 256, 256, 0, s>>>(G, nc, 1.0);
      CASPT2_CUDA_TRY(cudaGetLastError());
      CASPT2_CUDA_TRY(take_columns());
      const double lg = std::log2(std::max(1e-300, 0.5 * (double)m * dev_ortho));
      const int S = std::max(2, std::min(kOzMaxSlices, (int)std::ceil((57.0 + lg) / 7.0)));
      const int S0 = oz->S;
      oz->S = S;
      // G symmetric: B(j, k) = G[nc - nk + j][k]
      const OzView vz{Z, nc, 1, nc, 0}, vg{G + (long)(nc - nk) * nc, nc, 1, nc, 0};
      const cudaError_t e = oz_matmul(*oz, vz, vg, false, m, nk, nc, 1.0, 1.0, V, nk, s);
      oz->S = S0;
      CASPT2_CUDA_TRY(e);
    } else {
      CASPT2_CUDA_TRY(dgemm(m, nk, nc, 1.0, Z, nc, false, G + (nc - nk), nc, false, 0.0, V, nk, s));
    }
  }
  // 5. back-transformation V = H_0 ... H_{m-3} Z: blocked (compact WY panels as FP64
  //    GEMMs) for large matrices, else column-owned in one launch.  Z, G and the
  //    inverse-iteration scratch are free here.
  if (m >= kWyMinSize) {
    const int st = backtransform_wy(vbuf, tau, m, nk, V, Z, 7 * mm, s, oz);
    if (st != CASPT2_OK) return st;
  } else if (m >= 3) {
    // columns resident in shared memory: ceil(m / SMs) per block (one block per SM, the FP64
    // work spread evenly, one warp per column); below kWyMinSize rows 23 and more of them fit
    const int cbs = std::min(16, (nk + nsm - 1) / nsm);
    CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_backtransform_smem,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kBackSmemMax));
    ++launch_counter();
    k_backtransform_smem<<<(nk + cbs - 1) / cbs, 32 * cbs,
                           sizeof(double) * (size_t)m * (cbs + 2), s>>>(vbuf, tau, m, nk, cbs, V);
  }
  CASPT2_CUDA_TRY(cudaGetLastError());
  return CASPT2_OK;
}

}  // namespace caspt2
