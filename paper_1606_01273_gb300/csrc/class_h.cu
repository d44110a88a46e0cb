// Class H (E_ai,bj, Eq. class) of the first-order amplitudes, FP64, direct.
//
// For block-diagonal f the E_ai,bj E_Omega|N~> functions couple to the
// reference index only through the active Fock matrix: with U^T Fref U =
// W diag(omega) W^T, the amplitude equation (Eq. ampeq) for state L becomes, in
// the eigenbasis nu, a closed-shell pair equation with denominator
//     D = e_a + e_b - e_i - e_j + omega_nu - E0_L + E_s.
// The contributions to the effective Hamiltonian (Sec. II.B) are then
//     <Psi1_L|H|L'~>_H = -sum_nu W_Lnu W_L'nu sum_ijab K(2K - K')/D
//     <Psi1_L|Psi1_L>_H =  sum_nu W_Lnu^2     sum_ijab K(2K - K')/D^2
// with K = (ai|bj) = sum_P B_Pai B_Pbj, K' = (aj|bi).  Under SS-SR (Eq. wfp2) only
// nu = L survives and D = e_a + e_b - e_i - e_j + E_s.
//
// The amplitudes are never stored: one CTA forms a 64x64 tile of K_ij (and the
// mirrored tile) over the DF index, and the epilogue applies every
// denominator shift and reduces the energy and norm sums.  Per-CTA partial
// sums are reduced afterwards in a fixed order, so results are bitwise
// reproducible run to run.
#include "kernels.cuh"
#include "class_ag.cuh"
#include "ozaki.cuh"

namespace caspt2 {

constexpr int kHT = 64;   // tile edge in a and in b
constexpr int kHK = 16;   // DF-index chunk
constexpr int kHThreads = 256;
constexpr int kMaxShift = kMaxStates * kMaxStates;

// Bp[i][P][a] = B[P][i][vo + a]; go: nothing is done where it points to zero
__global__ void k_pack_cv(const double* __restrict__ B, int c, int v, int X, int nmo, int vo,
                          double* __restrict__ Bp, const int* __restrict__ go) {
  if (go && *go == 0) return;
  long total = (long)c * X * v;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total;
       idx += (long)gridDim.x * blockDim.x) {
    int a = idx % v;
    long iP = idx / v;
    int P = iP % X;
    int i = iP / X;
    Bp[idx] = B[((long)P * nmo + i) * nmo + vo + a];
  }
}

// eps[0..c) = closed orbital energies, eps[c..c+v) = virtual orbital energies
__global__ void k_eps_cv(const double* __restrict__ f, int nmo, int c, int a, int v, double* eps) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x < c) eps[x] = f[(long)x * nmo + x];
  else if (x < c + v) eps[x] = f[(long)(x + a) * nmo + x + a];
}

// shifts[nu*n + L] = omega_nu - E0_L + E_s (MS-MR) ; shifts[0] = E_s (SS-SR)
__global__ void k_classH_shifts(const double* __restrict__ omega, const double* __restrict__ E0,
                                double shift, int n, int scheme, double* shifts) {
  int k = threadIdx.x;
  if (scheme == CASPT2_SSSR) {
    if (k == 0) shifts[0] = shift;
    return;
  }
  if (k < n * n) shifts[k] = omega[k / n] - E0[k % n] + shift;
}

// One CTA = (pair i <= j, tile pair ta <= tb).  It forms T1[a][b] = K_ij^ab over
// a in tile ta, b in tile tb and, when ta < tb, T2[a][b] = K_ij^ba = sum_P B_ib B_ja,
// so each thread holds both K_ij^ab and K_ij^ba for its elements and the K_ij block
// is computed exactly once.  On a diagonal tile (ta == tb) K_ij^ba is read from the
// transposed tile staged in shared memory.  Block (j, i) equals block (i, j) with a
// and b swapped, so i < j carries weight 2; for i == j, K_ii^ba = K_ii^ab.  go: as in k_pack_cv.
__global__ void __launch_bounds__(kHThreads)
k_classH(const double* __restrict__ Bp, const double* __restrict__ eps,
         const double* __restrict__ shifts, int nshift, int c, int v, int X, int ntile,
         int pair0, double* __restrict__ partial, const int* __restrict__ go) {
  if (go && *go == 0) return;
  __shared__ double sbuf[4 * kHK * kHT];   // operand tiles; reused for the diagonal transpose
  __shared__ double sEa[kHT], sEb[kHT];
  __shared__ double sShift[kMaxShift];
  __shared__ double red[32];
  double (*sAi)[kHT] = reinterpret_cast<double (*)[kHT]>(sbuf);
  double (*sBj)[kHT] = reinterpret_cast<double (*)[kHT]>(sbuf + kHK * kHT);
  double (*sAj)[kHT] = reinterpret_cast<double (*)[kHT]>(sbuf + 2 * kHK * kHT);
  double (*sBi)[kHT] = reinterpret_cast<double (*)[kHT]>(sbuf + 3 * kHK * kHT);

  const int ntp = ntile * (ntile + 1) / 2;
  long bid = blockIdx.x;
  int tp = bid % ntp;
  int pair = pair0 + (int)(bid / ntp), i = 0;
  while (pair >= c - i) { pair -= c - i; ++i; }
  const int j = i + pair;
  int ta = 0;
  while (tp >= ntile - ta) { tp -= ntile - ta; ++ta; }
  const int tb = ta + tp;
  const bool same = (i == j);
  const bool diag = (ta == tb);
  const bool need_t2 = !same && !diag;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int a0 = ta * kHT, b0 = tb * kHT;
  const double* bi = Bp + (long)i * X * v;
  const double* bj = Bp + (long)j * X * v;

  for (int k = threadIdx.x; k < nshift; k += kHThreads) sShift[k] = shifts[k];
  for (int k = threadIdx.x; k < kHT; k += kHThreads) {
    sEa[k] = (a0 + k < v) ? eps[c + a0 + k] : 0.0;   // eps holds closed then virtual energies
    sEb[k] = (b0 + k < v) ? eps[c + b0 + k] : 0.0;
  }
  __syncthreads();

  double t1[4][4], t2[4][4];
#pragma unroll
  for (int ii = 0; ii < 4; ++ii)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) t1[ii][jj] = t2[ii][jj] = 0.0;

  for (int P0 = 0; P0 < X; P0 += kHK) {
    for (int l = threadIdx.x; l < kHK * kHT; l += kHThreads) {
      const int kk = l / kHT, col = l % kHT;
      const int P = P0 + kk;
      const bool okP = P < X;
      const int a = a0 + col, b = b0 + col;
      sAi[kk][col] = (okP && a < v) ? bi[(long)P * v + a] : 0.0;
      sBj[kk][col] = (okP && b < v) ? bj[(long)P * v + b] : 0.0;
      if (need_t2) {
        sAj[kk][col] = (okP && a < v) ? bj[(long)P * v + a] : 0.0;
        sBi[kk][col] = (okP && b < v) ? bi[(long)P * v + b] : 0.0;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kHK; ++kk) {
      double ra[4], rb[4];
#pragma unroll
      for (int ii = 0; ii < 4; ++ii) ra[ii] = sAi[kk][ty + 16 * ii];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) rb[jj] = sBj[kk][tx + 16 * jj];
#pragma unroll
      for (int ii = 0; ii < 4; ++ii)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) t1[ii][jj] = fma(ra[ii], rb[jj], t1[ii][jj]);
      if (need_t2) {
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) ra[ii] = sAj[kk][ty + 16 * ii];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) rb[jj] = sBi[kk][tx + 16 * jj];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) t2[ii][jj] = fma(ra[ii], rb[jj], t2[ii][jj]);
      }
    }
    __syncthreads();
  }

  if (same) {
#pragma unroll
    for (int ii = 0; ii < 4; ++ii)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) t2[ii][jj] = t1[ii][jj];
  } else if (diag) {
    // K_ij^ba of this thread's (a, b) is T1 at (b, a): stage T1 (64 x 64) and read it transposed
    double* sT = sbuf;
#pragma unroll
    for (int ii = 0; ii < 4; ++ii)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) sT[(ty + 16 * ii) * kHT + tx + 16 * jj] = t1[ii][jj];
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < 4; ++ii)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) t2[ii][jj] = sT[(tx + 16 * jj) * kHT + ty + 16 * ii];
  }

  // epilogue: numerators and shift-free denominators of this thread's 16 (a, b)
  const double wij = same ? 1.0 : 2.0;
  const double ei = eps[i], ej = eps[j];
  double num[16], d0[16];
#pragma unroll
  for (int ii = 0; ii < 4; ++ii)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int la = ty + 16 * ii, lb = tx + 16 * jj;
      const bool ok = (a0 + la < v) && (b0 + lb < v);
      const double k1 = t1[ii][jj];          // K_ij^ab
      const double k2 = t2[ii][jj];          // K_ij^ba
      // element (a, b); when ta < tb also element (b, a), which lives in no other CTA
      double nm = k1 * (2.0 * k1 - k2);
      if (!diag) nm += k2 * (2.0 * k2 - k1);
      num[ii * 4 + jj] = ok ? wij * nm : 0.0;
      d0[ii * 4 + jj] = ok ? (sEa[la] + sEb[lb] - ei - ej) : 1.0;
    }
  double* out = partial + blockIdx.x * (long)(3 * nshift + 1);
  double dmin = 1e300;
  for (int k = 0; k < nshift; ++k) {
    const double sh = sShift[k];
    double e = 0.0, nr = 0.0, n3 = 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const double inv = 1.0 / (d0[q] + sh);
      const double x = num[q] * inv;
      e += x;
      nr = fma(x, inv, nr);
      n3 = fma(x * inv, inv, n3);
      if (num[q] != 0.0) dmin = fmin(dmin, fabs(d0[q] + sh));
    }
    e = block_sum(e, red);
    if (threadIdx.x == 0) out[k] = e;
    nr = block_sum(nr, red);
    if (threadIdx.x == 0) out[nshift + k] = nr;
    n3 = block_sum(n3, red);
    if (threadIdx.x == 0) out[2 * nshift + k] = n3;
  }
  dmin = block_min(dmin, red);
  if (threadIdx.x == 0) out[3 * nshift] = dmin;
}

// sums[col] = fixed-order reduction of partial[.][col]; the last column is a min.  go: where it
// points to a nonzero, nblocks_go rows.
__global__ void k_reduce_cols(const double* __restrict__ partial, long nblocks, int ncol,
                              double* __restrict__ sums, const int* __restrict__ go = nullptr,
                              long nblocks_go = 0) {
  __shared__ double red[32];
  if (go && *go != 0) nblocks = nblocks_go;
  const int col = blockIdx.x;
  const bool is_min = (col == ncol - 1);
  double acc = is_min ? 1e300 : 0.0;
  for (long b = threadIdx.x; b < nblocks; b += blockDim.x) {
    double x = partial[b * ncol + col];
    acc = is_min ? fmin(acc, x) : acc + x;
  }
  acc = is_min ? block_min(acc, red) : block_sum(acc, red);
  if (threadIdx.x == 0) sums[col] = acc;
}

// Moments of class H from the sums Sk[nu,L] = sum num / D^k (k = 1, 2, 3):
//   M1[L][N][L'] = sum_nu W_Nnu W_L'nu S1[nu,L], M2[L][N] = sum_nu W_Nnu W_Lnu S2[nu,L],
//   M3[L] = sum_nu W_Lnu^2 S3[nu,L]; under SS-SR only N = L' = L with S_k[0].
// e[L][L'] = -M1[L][L][L'], norm[L] = M2[L][L].
__global__ void k_classH_combine(const double* __restrict__ sums, const double* __restrict__ W,
                                 int n, int scheme, double* ecls, double* ncls, double* mom,
                                 double* mindenom, int* status) {
  const int nshift = (scheme == CASPT2_SSSR) ? 1 : n * n;
  const double* S1 = sums;
  const double* S2 = sums + nshift;
  const double* S3 = sums + 2 * nshift;
  for (int idx = threadIdx.x; idx < n * n * n; idx += blockDim.x) {
    const int L = idx / (n * n), N = (idx / n) % n, Lp = idx % n;
    double v = 0.0;
    if (scheme == CASPT2_SSSR) v = (N == L && Lp == L) ? S1[0] : 0.0;
    else
      for (int nu = 0; nu < n; ++nu) v += W[N * n + nu] * W[Lp * n + nu] * S1[nu * n + L];
    mom[idx] = v;
    if (N == L) ecls[L * n + Lp] = -v;
  }
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int L = idx / n, N = idx % n;
    double v = 0.0;
    if (scheme == CASPT2_SSSR) v = (N == L) ? S2[0] : 0.0;
    else
      for (int nu = 0; nu < n; ++nu) v += W[N * n + nu] * W[L * n + nu] * S2[nu * n + L];
    mom[n * n * n + idx] = v;
    if (N == L) ncls[L] = v;
  }
  for (int L = threadIdx.x; L < n; L += blockDim.x) {
    double v = 0.0;
    if (scheme == CASPT2_SSSR) v = S3[0];
    else
      for (int nu = 0; nu < n; ++nu) v += W[L * n + nu] * W[L * n + nu] * S3[nu * n + L];
    mom[n * n * n + n * n + L] = v;
  }
  if (threadIdx.x == 0) {
    const double dm = sums[3 * nshift];
    *mindenom = fmin(*mindenom, dm);
    if (!(dm == dm)) atomicExch(status, CASPT2_ENAN);
  }
}

// Split form: KK[(ia)][(jb)] = K_ij^ab (2 K_ij^ab - K_ij^ba) from the full K matrix, j >= i
// (the sums below read no other).
__global__ void k_classH_num(const double* __restrict__ K, int c, int v, int i0, int i1,
                             double* __restrict__ KK) {
  const long cv = (long)c * v, e0 = (long)i0 * v * cv, total = (long)i1 * v * cv;
  for (long e = e0 + blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long ia = e / cv, jb = e % cv;
    const int i = ia / v, a = ia % v, j = jb / v, b = jb % v;
    if (j < i) continue;
    const double k1 = K[e];
    KK[e] = k1 * (2.0 * k1 - K[((long)i * v + b) * cv + (long)j * v + a]);
  }
}

// Split form: the sums of KK / D, KK / D^2, KK / D^3 over all (i, j, a, b) for G shifts of a
// block row (blockIdx.y) and the smallest |D| with KK != 0; one row of partial per block with
// only its own shifts' columns set (the others zero, the min column +inf for no element), so
// the fixed-order column reduction of the fused kernel applies unchanged.
//
// What bounds it: nine FP64 operations per element and shift (the reciprocal three, the three
// sums five, the denominator one) at two a clock and SM, 16 shifts for four states.  The
// elements (ia, jb) and (jb, ia) are equal (K and D are symmetric), so only jb >= ia is
// summed, off-diagonal ones twice; the G shifts of an element share its loads and give G
// independent chains.  c42 v350, 16 shifts: 82.9 ms with one shift a block over the full
// square.
// KK: element (ia, jb) at KK[ia * ld + jb - off].
template <int G>
__global__ void k_classH_sums(const double* __restrict__ KK, long ld, long off,
                              const double* __restrict__ eps, const double* __restrict__ shifts,
                              int nshift, int c, int v, int i0, int i1,
                              double* __restrict__ partial) {
  __shared__ double red[32];
  const int k0 = blockIdx.y * G;
  double sh[G], e[G], nr[G], n3[G];
  // smallest |D| with KK != 0, kept as the bit pattern of |D| (non-negative doubles order
  // like their bit patterns, so the minimum runs on the integer units)
  unsigned long long dminb = 0x7FF0000000000000ull;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    sh[g] = shifts[min(k0 + g, nshift - 1)];
    e[g] = nr[g] = n3[g] = 0.0;
  }
  // rows (i, a) over the blocks, (j, b) of a row over the threads: index arithmetic once
  // per row and per j, not per element
  for (long ia = (long)i0 * v + blockIdx.x; ia < (long)i1 * v; ia += gridDim.x) {
    const int i = (int)(ia / v), a = (int)(ia % v);
    const double base = eps[c + a] - eps[i];
    const double* row = KK + (ia * ld - off);
    for (int j = i; j < c; ++j) {
      const double bj = base - eps[j];
      const double* rj = row + (long)j * v;
      for (int b = (j == i ? a : 0) + threadIdx.x; b < v; b += blockDim.x) {
        double num = rj[b];
        if (j != i || b != a) num += num;
        const double D0 = bj + eps[c + b];
        const bool live = (__double_as_longlong(num) << 1) != 0;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const double D = D0 + sh[g];
          const double inv = recip(D);
          const double x = num * inv;
          e[g] += x;
          nr[g] = fma(x, inv, nr[g]);
          n3[g] = fma(x * inv, inv, n3[g]);
          const unsigned long long db =
              (unsigned long long)__double_as_longlong(D) & 0x7FFFFFFFFFFFFFFFull;
          if (live && db < dminb) dminb = db;
        }
      }
    }
  }
  double dmin = dminb < 0x7FF0000000000000ull ? __longlong_as_double((long long)dminb) : 1e300;
  const int ncol = 3 * nshift + 1;
  double* out = partial + ((long)blockIdx.y * gridDim.x + blockIdx.x) * ncol;
  for (int t = threadIdx.x; t < 3 * nshift; t += blockDim.x) out[t] = 0.0;
  __syncthreads();
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const double s1 = block_sum(e[g], red), s2 = block_sum(nr[g], red), s3 = block_sum(n3[g], red);
    if (threadIdx.x == 0 && k0 + g < nshift) {
      out[k0 + g] = s1;
      out[nshift + k0 + g] = s2;
      out[2 * nshift + k0 + g] = s3;
    }
  }
  dmin = block_min(dmin, red);
  if (threadIdx.x == 0) out[3 * nshift] = dmin;
}

cudaError_t launch_eps_cv(const double* f, const Dims& d, double* eps, cudaStream_t s) {
  if (d.c + d.v == 0) return cudaSuccess;
  ++launch_counter();
  k_eps_cv<<<(d.c + d.v + 127) / 128, 128, 0, s>>>(f, d.nmo(), d.c, d.a, d.v, eps);
  return cudaGetLastError();
}

long classH_blocks(const Dims& d) {
  long ntile = (d.v + kHT - 1) / kHT;
  long npair = (long)d.c * (d.c + 1) / 2;
  return npair * (ntile * (ntile + 1) / 2);
}

int classH_nshift(const Dims& d, int scheme) { return scheme == CASPT2_SSSR ? 1 : d.n * d.n; }

namespace {
// The pair sums of closed orbitals [i0, i1) by the fused kernel into the first `rows` rows of
// w.partial (go: only where it points to a nonzero).
cudaError_t launch_fused(const double* B, const Dims& d, int nshift, ClassHWork& w, int i0, int i1,
                         const int* go, long& rows, cudaStream_t s) {
  const int ntile = (d.v + kHT - 1) / kHT;
  // pairs (i <= j) with i in [i0, i1): a contiguous run of the row-major pair order
  auto start = [&](long i) { return i * d.c - i * (i - 1) / 2; };
  const long pair0 = start(i0), npair = start(i1) - start(i0);
  rows = npair * ((long)ntile * (ntile + 1) / 2);
  if (rows == 0) return cudaSuccess;
  const long tp = (long)d.c * d.X * d.v;
  ++launch_counter();
  k_pack_cv<<<(int)std::min<long>((tp + 255) / 256, 152 * 32), 256, 0, s>>>(
      B, d.c, d.v, d.X, d.nmo(), d.c + d.a, w.Bp, go);
  if (w.ev_gemm0 && !go) cudaEventRecord(w.ev_gemm0, s);
  ++launch_counter();
  k_classH<<<(unsigned)rows, kHThreads, 0, s>>>(w.Bp, w.eps, w.shifts, nshift, d.c, d.v, d.X,
                                               ntile, (int)pair0, w.partial, go);
  if (w.ev_gemm1 && !go) cudaEventRecord(w.ev_gemm1, s);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_classH(const double* f, const double* B, const double* Ftil, const double* E0,
                          double shift, int scheme, const Dims& d, ClassHWork& w, int* status,
                          double* ecls, double* ncls, double* mom, double* mindenom,
                          cudaStream_t s, int i0, int i1) {
  const int n = d.n, nmo = d.nmo();
  const int nshift = classH_nshift(d, scheme);
  cudaError_t e;
  if (d.c == 0 || d.v == 0) {
    e = cudaMemsetAsync(ecls, 0, sizeof(double) * n * n, s);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(ncls, 0, sizeof(double) * n, s);
  }
  ++launch_counter();
  k_eps_cv<<<(d.c + d.v + 127) / 128, 128, 0, s>>>(f, nmo, d.c, d.a, d.v, w.eps);
  e = launch_sym_eig(Ftil, n, w.W, w.omega, 0, status, s);
  if (e != cudaSuccess) return e;
  ++launch_counter();
  k_classH_shifts<<<1, kMaxShift, 0, s>>>(w.omega, E0, shift, n, scheme, w.shifts);
  if (i1 < 0 || i1 > d.c) i1 = d.c;
  long nb = 0;
  if ((e = launch_fused(B, d, nshift, w, i0, i1, nullptr, nb, s)) != cudaSuccess) return e;
  if (nb == 0) {
    e = cudaMemsetAsync(ecls, 0, sizeof(double) * n * n, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(mom, 0, sizeof(double) * (n * n * n + n * n + n), s);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(ncls, 0, sizeof(double) * n, s);
  }
  const int ncol = 3 * nshift + 1;
  ++launch_counter();
  k_reduce_cols<<<ncol, 256, 0, s>>>(w.partial, nb, ncol, w.sums);
  ++launch_counter();
  k_classH_combine<<<1, 256, 0, s>>>(w.sums, w.W, n, scheme, ecls, ncls, mom, mindenom, status);
  return cudaGetLastError();
}

namespace {
// Shifts per block row of k_classH_sums: the group of three to five that pads nshift least (one
// shift: one).
int shift_group(int nshift) {
  if (nshift <= 1) return 1;
  int G = 4;
  for (int g : {5, 3})
    if ((nshift + g - 1) / g * g < (nshift + G - 1) / G * G) G = g;
  return G;
}

void launch_sums(int G, int nblk, const double* KK, long ld, long off, const ClassHWork& w,
                 int nshift, const Dims& d, int i0, int i1, double* partial, cudaStream_t s) {
  const dim3 grid(nblk, (nshift + G - 1) / G);
  // one pass over b per (i, a, j) when v fits a block (no idle tail of lanes)
  const int threads = d.v <= 512 ? std::max(64, (d.v + 31) / 32 * 32) : 256;
  auto run = [&](auto kernel) {
    kernel<<<grid, threads, 0, s>>>(KK, ld, off, w.eps, w.shifts, nshift, d.c, d.v, i0, i1,
                                    partial);
  };
  ++launch_counter();
  if (G == 1) run(k_classH_sums<1>);
  else if (G == 3) run(k_classH_sums<3>);
  else if (G == 4) run(k_classH_sums<4>);
  else run(k_classH_sums<5>);
}
}  // namespace

cudaError_t launch_classH_split(const double* f, const double* B, const double* Ftil,
                                const double* E0, double shift, int scheme, const Dims& d,
                                ClassHWork& w, int* status, double* ecls, double* ncls,
                                double* mom, double* mindenom, OzWork& oz, double* pack,
                                double* K, double* KK, cudaStream_t s, int i0, int i1) {
  const int n = d.n, nmo = d.nmo();
  const int nshift = classH_nshift(d, scheme);
  cudaError_t e;
  if (d.c == 0 || d.v == 0) {
    e = cudaMemsetAsync(ecls, 0, sizeof(double) * n * n, s);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(ncls, 0, sizeof(double) * n, s);
  }
  ++launch_counter();
  k_eps_cv<<<(d.c + d.v + 127) / 128, 128, 0, s>>>(f, nmo, d.c, d.a, d.v, w.eps);
  e = launch_sym_eig(Ftil, n, w.W, w.omega, 0, status, s);
  if (e != cudaSuccess) return e;
  ++launch_counter();
  k_classH_shifts<<<1, kMaxShift, 0, s>>>(w.omega, E0, shift, n, scheme, w.shifts);
  const long cv = (long)d.c * d.v;
  if (i1 < 0 || i1 > d.c) i1 = d.c;
  if (i1 <= i0) {
    e = cudaMemsetAsync(ecls, 0, sizeof(double) * n * n, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(mom, 0, sizeof(double) * (n * n * n + n * n + n), s);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(ncls, 0, sizeof(double) * n, s);
  }
  if ((e = launch_pack_block(B, d, SP_C, SP_V, pack, s)) != cudaSuccess) return e;
  if (w.ev_gemm0) cudaEventRecord(w.ev_gemm0, s);
  // rows (ia) with i in [i0, i1) of K = Bcv^T Bcv (the whole K for the full range); the
  // exchange partner K(aj|bi) = K(bi|aj) lies in the same rows
  const long r0 = (long)i0 * d.v, nr = (long)(i1 - i0) * d.v;
  const OzView vp{pack, 1, cv, (long)d.X, 0};     // rows (ia), K = Q
  const OzView vr{pack + r0, 1, cv, (long)d.X, 0};
  if (nr == cv) {
    if ((e = oz_matmul(oz, vp, vp, true, (int)cv, (int)cv, d.X, 1.0, 0.0, K, cv, s)) != cudaSuccess)
      return e;
  } else if ((e = oz_matmul(oz, vr, vp, false, (int)nr, (int)cv, d.X, 1.0, 0.0, K + r0 * cv, cv,
                            s)) != cudaSuccess) {
    return e;
  }
  if (w.ev_gemm1) cudaEventRecord(w.ev_gemm1, s);
  const long total = nr * cv;
  ++launch_counter();
  k_classH_num<<<(int)std::min<long>((total + 255) / 256, 152L * 32), 256, 0, s>>>(K, d.c, d.v, i0,
                                                                                  i1, KK);
  const int G = shift_group(nshift), ng = (nshift + G - 1) / G;
  const int nblk = (int)std::max<long>(1, std::min<long>(w.nblocks / ng, 152L * 8));
  launch_sums(G, nblk, KK, cv, 0, w, nshift, d, i0, i1, w.partial, s);
  const int ncol = 3 * nshift + 1;
  ++launch_counter();
  k_reduce_cols<<<ncol, 256, 0, s>>>(w.partial, (long)nblk * ng, ncol, w.sums);
  ++launch_counter();
  k_classH_combine<<<1, 256, 0, s>>>(w.sums, w.W, n, scheme, ecls, ncls, mom, mindenom, status);
  return cudaGetLastError();
}

// In place: K_ij^ab -> K_ij^ab (2 K_ij^ab - K_ij^ba) for i in [i0, i0 + ni), j >= i0; element
// (ia, jb) at K[(ia - i0 v) ld + jb - i0 v].  Both 32 x 32 tiles of a pair (a, b), (b, a) go through
// shared memory, so that all global accesses run along b (c42 v350: the transposed read of
// k_classH_num costs 1.27 ms where the bytes take 0.4).  grid (tile pairs ta <= tb, (i, j)).
__global__ void __launch_bounds__(256)
k_classH_num_tiles(double* __restrict__ K, long ld, int v, int ni, int nj) {
  __shared__ double t1[32][33], t2[32][33];
  const int nt = (v + 31) / 32;
  int ta = 0, rem = blockIdx.x;
  while (rem >= nt - ta) { rem -= nt - ta; ++ta; }
  const int a0 = 32 * ta, b0 = 32 * (ta + rem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long ij = blockIdx.y; ij < (long)ni * nj; ij += gridDim.y) {
    const int i = (int)(ij / nj), j = (int)(ij % nj);
    if (j < i) continue;                       // the same for the whole block
    double* base = K + (long)i * v * ld + (long)j * v;
    for (int r = warp; r < 32; r += 8) {
      t1[r][lane] = a0 + r < v && b0 + lane < v ? base[(a0 + r) * ld + b0 + lane] : 0.0;
      t2[r][lane] = b0 + r < v && a0 + lane < v ? base[(b0 + r) * ld + a0 + lane] : 0.0;
    }
    __syncthreads();
    for (int r = warp; r < 32; r += 8) {
      const double x = t1[r][lane], y = t2[r][lane];
      if (a0 + r < v && b0 + lane < v) base[(a0 + r) * ld + b0 + lane] = x * (2.0 * x - t2[lane][r]);
      if (a0 != b0 && b0 + r < v && a0 + lane < v)
        base[(b0 + r) * ld + a0 + lane] = y * (2.0 * y - t1[lane][r]);
    }
    __syncthreads();
  }
}

// What the slices may cost, checked on the data of every solve.  An element of K from eight
// slices is off by up to 1.13 2^-55 X s_ia s_jb (kOzFp64Slices; s: row scales), whatever its size, one
// from FP64 fused multiply-adds by up to 2^-53 X sum_P |B_P,ia B_P,jb|, which is at least
// 2^-53 X |K|.  To first order a returned sum O = sum_ijab w K (2K - K'), w = |D|^-p, moves by
// sum w |K| (4 s_ia s_jb + 2 s_ib s_ja) times the element's error, so slicing costs O no more than
// FP64 products may where
//   g = 0.29 |K| (4 s_ia s_jb + 2 s_ib s_ja) + c2 (s_ia s_jb)^2 - 4 K^2
// (c2 = 1.3 2^-55 X: the second order) has sum w g <= 0 for every shift and p = 1, 2, 3.  It holds by
// a factor of 4 to 40 for factors of evenly sized elements, by 2 to 7 for local orbitals, and by 1.2
// for elements that fall by e^20 over P, and fails where the pairs that matter have their large
// elements at different P (rows graded in opposite directions and a range of closed orbitals whose
// own pairs are small): those solves take the fused kernel.
// FP32 throughout (the units are idle and the sum's sign is far from its rounding): s as multiples
// of the largest among the rows i, and among the rows j, of the call; K from the bits of its upper
// word.  One pass over K.
__global__ void __launch_bounds__(1024)
k_guard_scale(const double* __restrict__ sc, const double* __restrict__ eps, int r0, int r1, int cv,
              int ne, float* __restrict__ sgi, float* __restrict__ sgj, float* __restrict__ ef,
              int* __restrict__ es) {
  __shared__ int red[2][32];
  // largest exponent fields (the scales are powers of two, 0 or NaN) over [r0, r1) and [r0, cv)
  int mi = 1, mj = 1;
  for (int r = r0 + threadIdx.x; r < cv; r += blockDim.x) {
    const int b = __double2hiint(sc[r]) >> 20;
    if (b >= 2047) continue;
    mj = max(mj, b);
    if (r < r1) mi = max(mi, b);
  }
  mi = __reduce_max_sync(0xffffffffu, mi);
  mj = __reduce_max_sync(0xffffffffu, mj);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = mi;
    red[1][threadIdx.x >> 5] = mj;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    mi = __reduce_max_sync(0xffffffffu, red[0][threadIdx.x]);
    mj = __reduce_max_sync(0xffffffffu, red[1][threadIdx.x]);
    if (threadIdx.x == 0) {
      red[0][0] = mi;
      red[1][0] = mj;
      *es = mi + mj - 2046;
    }
  }
  __syncthreads();
  mi = red[0][0];
  mj = red[1][0];
  for (int r = threadIdx.x; r < cv; r += blockDim.x) {
    const int b = __double2hiint(sc[r]) >> 20;
    sgi[r] = b == 0 ? 0.f : b == 2047 ? nanf("") : exp2f((float)(b - mi));
    sgj[r] = b == 0 ? 0.f : b == 2047 ? nanf("") : exp2f((float)(b - mj));
  }
  for (int k = threadIdx.x; k < ne; k += blockDim.x) ef[k] = (float)eps[k];
}

// Grid as k_classH_sums; out[((block) ng + group) 3G + 3 g + p - 1].
template <int G>
__global__ void k_classH_guard(const double* __restrict__ K, long ld, long off,
                               const float* __restrict__ sgi, const float* __restrict__ sgj,
                               const float* __restrict__ ef, const int* __restrict__ es,
                               const double* __restrict__ shifts, int nshift, int c, int v, int i0, int i1, float c2,
                               double* __restrict__ out) {
  __shared__ double red[32];
  const int k0 = blockIdx.y * G, e2 = *es;
  float sh[G], a1[G], a2[G], a3[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    sh[g] = (float)shifts[min(k0 + g, nshift - 1)];
    a1[g] = a2[g] = a3[g] = 0.f;
  }
  for (long ia = (long)i0 * v + blockIdx.x; ia < (long)i1 * v; ia += gridDim.x) {
    const int i = (int)(ia / v), a = (int)(ia % v);
    const float base = ef[c + a] - ef[i], sia = sgi[ia];
    const double* row = K + (ia * ld - off);
    for (int j = i; j < c; ++j) {
      const float bj = base - ef[j], sja = sgj[(long)j * v + a];
      const double* rj = row + (long)j * v;
      for (int b = (j == i ? a : 0) + threadIdx.x; b < v; b += blockDim.x) {
        // |K| / (s_max s_max') from the upper word: exponent field moved, 20 bits of the significand
        const unsigned hi = (unsigned)__double2hiint(rj[b]) & 0x7FFFFFFFu;
        const int ex = (int)(hi >> 20);
        const int fx = ex == 2047 ? 255 : max(0, min(254, ex - 1023 - e2 + 127));
        const float k = fx == 0 || ex == 0 ? 0.f
                        : __uint_as_float((unsigned)fx << 23 | (hi & 0xFFFFFu) << 3 | (ex == 2047));
        const float s1 = sia * sgj[(long)j * v + b], s2 = sgi[(long)i * v + b] * sja;
        float q = fmaf(k, 0.29f * fmaf(4.f, s1, 2.f * s2), fmaf(c2 * s1, s1, -4.f * k * k));
        if (j != i || b != a) q += q;
        const float D0 = bj + ef[c + b];
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float w = __fdividef(1.f, fabsf(D0 + sh[g])), x = q * w, y = x * w;
          a1[g] += x;
          a2[g] += y;
          a3[g] = fmaf(y, w, a3[g]);
        }
      }
    }
  }
  double* o = out + ((long)blockIdx.x * gridDim.y + blockIdx.y) * (3 * G);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const double t1 = block_sum((double)a1[g], red), t2 = block_sum((double)a2[g], red),
                 t3 = block_sum((double)a3[g], red);
    if (threadIdx.x == 0) {
      o[3 * g] = t1;
      o[3 * g + 1] = t2;
      o[3 * g + 2] = t3;
    }
  }
}

// *go = 1 where a column's sum over the rows is above zero or not a number; a block a column.
__global__ void k_guard_decide(const double* __restrict__ part, long rows, int ncol,
                               int* __restrict__ go) {
  __shared__ double red[32];
  double s = 0.0;
  for (long r = threadIdx.x; r < rows; r += blockDim.x) s += part[r * ncol + blockIdx.x];
  s = block_sum(s, red);
  if (threadIdx.x == 0 && !(s <= 0.0)) *go = 1;
}

namespace {
int sliced_rows(const Dims& d, int i, long cap) {   // closed orbitals of the chunk from i on
  return (int)std::min<long>(d.c - i, cap / ((long)d.v * (d.c - i) * d.v));
}
int sliced_chunks(const Dims& d, long kcap) {
  int n = 0;
  for (int i = 0; i < d.c; i += sliced_rows(d, i, kcap)) ++n;
  return n;
}
}  // namespace

// Doubles of the K workspace, or 0 where the fused kernel serves: up to 2^26 multiply-adds of the
// full product, where it takes 0.16 (c4 v20 X84), 0.34 (c4 v64 X256) and 0.6 ms (c4 v128 X256) of a
// pass of 4 ms or more and needs neither workspace nor a bound on its error; slices would take
// 0.11, 0.13 and 0.14.  Just above the line 0.70 against 0.15 (c6 v90 X300).  The workspace is one
// chunk of rows, 128 MB unless a single closed orbital needs more.
long classH_sliced_work(const Dims& d, int scheme) {
  const double cv = (double)d.c * d.v, fmas = cv * cv * d.X;
  if (fmas <= 67108864.0 || d.X > (1 << 17) || cv > 1e9) return 0;
  return std::min<long>((long)(cv * cv), std::max<long>(1L << 24, (long)(cv * d.v)));
}

// Rows of the partial sums: a block's each in the fused kernel; the split forms take up to
// eight blocks a SM and shift group (c8 v61, nine shifts: the fused kernel's 36 rows left 12 blocks a
// group, 0.27 ms), in at most 64 MB.
long classH_partial_rows(const Dims& d, int scheme, bool split) {
  const long kcap = split ? (long)d.c * d.v * d.c * d.v : classH_sliced_work(d, scheme);
  if (kcap <= 0) return classH_blocks(d);
  const int nshift = classH_nshift(d, scheme), G = shift_group(nshift);
  const long chunks = sliced_chunks(d, kcap);
  const long per = chunks * ((nshift + G - 1) / G);
  const long nblk = std::min({152L * 8, (long)d.c * d.v, (1L << 23) / (per * (3 * nshift + 1))});
  return std::max(classH_blocks(d), per * std::max(1L, nblk));
}

namespace {
constexpr int kGuardBlocks = 152 * 4;                // of a chunk and shift group

// The guard's arrays in w.guard: partial sums, then row scales and orbital energies in FP32, the
// scales' exponent and the decision.
struct GuardArrays {
  double* part;
  float *sgi, *sgj, *ef;
  int *es, *go;
};
size_t guard_part(const Dims& d, int scheme) {
  const int nshift = classH_nshift(d, scheme), G = shift_group(nshift);
  return (size_t)sliced_chunks(d, classH_sliced_work(d, scheme)) * kGuardBlocks *
         ((nshift + G - 1) / G) * 3 * G;
}
GuardArrays guard_arrays(const Dims& d, int scheme, double* g) {
  GuardArrays a;
  a.part = g;
  a.sgi = reinterpret_cast<float*>(g + guard_part(d, scheme));
  a.sgj = a.sgi + (size_t)d.c * d.v;
  a.ef = a.sgj + (size_t)d.c * d.v;
  a.es = reinterpret_cast<int*>(a.ef + d.c + d.v);
  a.go = a.es + 1;
  return a;
}
}  // namespace

size_t classH_guard_size(const Dims& d, int scheme) {
  return guard_part(d, scheme) + (2 * (size_t)d.c * d.v + d.c + d.v + 2 + 1) / 2;
}

cudaError_t classH_sliced_reserve(const Dims& d, OzWork& oz) {
  const int cv = d.c * d.v;
  return oz_reserve(oz, oz_slice_bytes(cv, d.X, kOzFp64Slices), cv);
}

namespace {
void launch_guard(int G, const double* K, long ld, long off, const ClassHWork& w,
                  const GuardArrays& ga, int nshift, const Dims& d, int i0, int i1, float c2,
                  long at, cudaStream_t s) {
  const dim3 grid(kGuardBlocks, (nshift + G - 1) / G);
  const int threads = d.v <= 512 ? std::max(64, (d.v + 31) / 32 * 32) : 256;
  auto run = [&](auto kernel) {
    kernel<<<grid, threads, 0, s>>>(K, ld, off, ga.sgi, ga.sgj, ga.ef, ga.es, w.shifts, nshift,
                                    d.c, d.v, i0, i1, c2, ga.part + at);
  };
  ++launch_counter();
  if (G == 1) run(k_classH_guard<1>);
  else if (G == 3) run(k_classH_guard<3>);
  else if (G == 4) run(k_classH_guard<4>);
  else run(k_classH_guard<5>);
}
}  // namespace

// Plain form at sizes where the FP64 units decide (classH_sliced_work): the products of
// k_classH as exact BF16 slices on the tensor cores, eight an operand.  B_cv is sliced once; chunks
// of closed orbitals i form K for their rows and j >= i in a bounded workspace, the numerators in
// its place and the sums.  Where k_guard_decide finds that the slices may cost a returned sum
// more than FP64 products do, the fused kernel forms the sums instead (its launches return at once
// otherwise, so the host need not wait for the decision).
// c30 v300 X990, a pass with inputs: 77.7 ms fused (the FMAs alone take 69), 7.9 here: GEMMs 5.0,
// sums 1.2, numerators 0.3, guard 0.25, slicing 0.15, inputs 0.3; the energies' error against 64 bits
// 2.7e-16.
cudaError_t launch_classH_sliced(const double* f, const double* B, const double* Ftil,
                                 const double* E0, double shift, int scheme, const Dims& d,
                                 ClassHWork& w, int* status, double* ecls, double* ncls,
                                 double* mom, double* mindenom, OzWork& oz, double* K, long kcap,
                                 cudaStream_t s, int i0, int i1) {
  const int n = d.n, nshift = classH_nshift(d, scheme);
  if (i1 < 0 || i1 > d.c) i1 = d.c;
  cudaError_t e;
  if (i1 <= i0) {
    if ((e = cudaMemsetAsync(ecls, 0, sizeof(double) * n * n, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(mom, 0, sizeof(double) * (n * n * n + n * n + n), s)) != cudaSuccess)
      return e;
    return cudaMemsetAsync(ncls, 0, sizeof(double) * n, s);
  }
  if ((e = launch_eps_cv(f, d, w.eps, s)) != cudaSuccess) return e;
  if ((e = launch_sym_eig(Ftil, n, w.W, w.omega, 0, status, s)) != cudaSuccess) return e;
  ++launch_counter();
  k_classH_shifts<<<1, kMaxShift, 0, s>>>(w.omega, E0, shift, n, scheme, w.shifts);
  if ((e = launch_pack_block(B, d, SP_C, SP_V, w.Bp, s)) != cudaSuccess) return e;
  if (w.ev_gemm0) cudaEventRecord(w.ev_gemm0, s);
  const int cv = d.c * d.v, Kp = oz_kpad(d.X), S = kOzFp64Slices;
  if ((e = classH_sliced_reserve(d, oz)) != cudaSuccess) return e;
  const OzView vb{w.Bp, 1, cv, (long)d.X, 0};        // rows (ia), K = P
  if ((e = oz_split(vb, cv, d.X, Kp, S, oz.sl, oz.sc, s)) != cudaSuccess) return e;
  const long plane = (long)cv * Kp;
  const int chunks = sliced_chunks(d, kcap);
  const GuardArrays ga = guard_arrays(d, scheme, w.guard);
  if ((e = cudaMemsetAsync(ga.go, 0, sizeof(int), s)) != cudaSuccess) return e;
  ++launch_counter();
  k_guard_scale<<<1, 1024, 0, s>>>(oz.sc, w.eps, i0 * d.v, i1 * d.v, cv, d.c + d.v, ga.sgi, ga.sgj,
                                   ga.ef, ga.es);
  const float c2 = (float)(1.3 * 0x1p-55 * d.X);
  const int G = shift_group(nshift), ng = (nshift + G - 1) / G, ncol = 3 * nshift + 1;
  const int nblk = (int)std::max<long>(1, std::min<long>(w.nblocks / ((long)ng * chunks), 152L * 8));
  long used = 0, gused = 0;
  const int nt = (d.v + 31) / 32;
  for (int i = i0; i < i1;) {
    const int ni = std::min(sliced_rows(d, i, kcap), i1 - i), nj = d.c - i;
    const long r0 = (long)i * d.v;
    const int M = ni * d.v, N = nj * d.v;
    const __nv_bfloat16* sl = oz.sl + r0 * Kp;
    if ((e = oz_gemm(sl, oz.sc + r0, sl, oz.sc + r0, M, N, Kp, S, 1.0, 0.0, K, N, oz.err, s, 1,
                     nullptr, false, plane, plane)) != cudaSuccess)
      return e;
    launch_guard(G, K, N, r0 * N + r0, w, ga, nshift, d, i, i + ni, c2, gused * ng * 3 * G, s);
    gused += kGuardBlocks;
    ++launch_counter();
    k_classH_num_tiles<<<dim3(nt * (nt + 1) / 2, std::min(ni * nj, 65535)), 256, 0, s>>>(K, N, d.v,
                                                                                        ni, nj);
    launch_sums(G, nblk, K, N, r0 * N + r0, w, nshift, d, i, i + ni, w.partial + used * ncol, s);
    used += (long)nblk * ng;
    i += ni;
  }
  ++launch_counter();
  k_guard_decide<<<ng * 3 * G, 256, 0, s>>>(ga.part, gused, ng * 3 * G, ga.go);
  long fused = 0;
  if ((e = launch_fused(B, d, nshift, w, i0, i1, ga.go, fused, s)) != cudaSuccess) return e;
  if (w.ev_gemm1) cudaEventRecord(w.ev_gemm1, s);
  ++launch_counter();
  k_reduce_cols<<<ncol, 256, 0, s>>>(w.partial, used, ncol, w.sums, ga.go, fused);
  ++launch_counter();
  k_classH_combine<<<1, 256, 0, s>>>(w.sums, w.W, n, scheme, ecls, ncls, mom, mindenom, status);
  return cudaGetLastError();
}

}  // namespace caspt2
