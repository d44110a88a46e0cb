// Classes A-G: the class share of the correlated densities of a target state P
// (Sec. II.D) from the sector bases kept by the energy pass.
//
// With R the eigenvectors of H^eff, r = R[:, P], and T_L, lambda_L the first-order
// amplitudes and the lambda amplitudes (Eq. lambdaeq) over all index tuples,
//   W_L'   = r_L' sum_L r_L T_L + lambda_L'                (source multiplier)
//   d1_pq  = sum W <M~|E_Omega^dag E_pq|L'~>                (d/dh of the sources)
//   G_pqrt = sum W <M~|E_Omega^dag 1/2 E_pq,rt|L'~>         (d/d(pq|rt))
//   d2     = d L / d f on the closed, active and virtual blocks:
//            closed/virtual: one external slot of T moves (hole or particle line of
//            f), contracted through the overlap (identity or pair swap);
//            active: lambda x T contracted with the d/df_uw of F_act, minus
//            N_L <L~|E_uw|L~> from the E0 dependence of the denominators.
// All contractions reuse the access plans of the solve (transposed), so the device
// path shares the solve's normal ordering and index conventions.
#include <cmath>
#include <type_traits>
#include <vector>

#include "class_ag.cuh"
#include "class_dev.cuh"
#include "linalg.cuh"

namespace caspt2 {

namespace {

constexpr double kInvSqrt2 = 0.70710678118654752440;
constexpr long kActAdjSmem = 96L * 1024;

// Sector amplitudes and lambda in the eigenbasis mu of the sector, for every
// (tuple t, state L): amp = -Vt_L / D_L, lam = -(r_L sum_N r_N Vt_N - 2 E_s r_L^2 amp) / D_L,
// D_L = e_ext(t) + omega_mu - E0_L + E_s.  Layout [mu][t][Li] (Li = L, or 0 for SS-SR).
__global__ void k_sector_amp(const double* __restrict__ Vt, const double* __restrict__ omega,
                             const double* __restrict__ E0, const double* __restrict__ eps,
                             const double* __restrict__ R, int P, DevClass C, ExtDims ed, int c,
                             int n, int sector, int Lsel, long ntup, int nk, double shift,
                             double* __restrict__ amp, double* __restrict__ lam) {
  const int nL = Lsel < 0 ? n : 1;
  const long ncolV = ntup * n;
  const long total = (long)nk * ntup * nL;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const int Li = e % nL;
    const long t = (e / nL) % ntup;
    const long mu = e / (nL * ntup);
    const int L = Lsel < 0 ? Li : Lsel;
    int co[3], cs[3];
    sector_tuple(C, ed.d, sector, t, co, cs);
    double ee = 0.0;
    for (int k = 0; k < C.next; ++k)
      ee += (C.slot_space[C.ext[k]] == SP_V) ? eps[c + co[k]] : -eps[co[k]];
    const double D = ee + omega[mu] - E0[L] + shift;
    const double* row = Vt + mu * ncolV + t * n;
    const double am = -row[L] / D;
    double acc = 0.0;
    for (int N = 0; N < n; ++N) acc += R[N * n + P] * row[N];
    const double rl = R[L * n + P];
    amp[e] = am;
    lam[e] = -(rl * acc - 2.0 * shift * rl * rl * am) / D;
  }
}

// Sector rows src[i][(t, Li)] (i over the sector rows) -> all-tuple arrays
// dst[tuple][L][row]; pair classes: a pair (x, y), x < y, receives (T+ + T-)/sqrt2 and its
// swap (T+ - T-)/sqrt2, x = y receives T+.  Two arrays (T and lambda) per launch.
__global__ void k_tuple_scatter(const double* __restrict__ src0, const double* __restrict__ src1,
                                DevClass C, ExtDims ed, int n, int m, int sector, int Lsel,
                                long ntup, int msec, double* __restrict__ dst0,
                                double* __restrict__ dst1) {
  const int nL = Lsel < 0 ? n : 1;
  const long ncol = ntup * nL;
  const long total = (long)msec * ncol;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long i = e / ncol, col = e % ncol;
    const long t = col / nL;
    const int Li = col % nL;
    const int L = Lsel < 0 ? Li : Lsel;
    const long row = Lsel < 0 ? i : i * n + Lsel;
    int co[3], cs[3];
    sector_tuple(C, ed.d, sector, t, co, cs);
    const long ia = (tuple_index(C, ed.d, co) * n + L) * m + row;
    const long ib = (tuple_index(C, ed.d, cs) * n + L) * m + row;
    const double x0 = src0[e], x1 = src1[e];
    if (C.pair0 < 0) {
      dst0[ia] = x0;
      dst1[ia] = x1;
    } else if (ia == ib) {
      dst0[ia] += x0;
      dst1[ia] += x1;
    } else {
      const double sg = sector == 0 ? kInvSqrt2 : -kInvSqrt2;
      dst0[ia] += kInvSqrt2 * x0;
      dst1[ia] += kInvSqrt2 * x1;
      dst0[ib] += sg * x0;
      dst1[ib] += sg * x1;
    }
  }
}

// dst[t][inner] = src[swap(t)][inner], swap exchanging the pair slots of the tuple.
__global__ void k_swap_tuples(const double* __restrict__ src, DevClass C, ExtDims ed, long ntot,
                              long inner, double* __restrict__ dst) {
  int ip = 0, jp = 0;
  for (int k = 0; k < C.next; ++k) {
    if (C.ext[k] == C.pair0) ip = k;
    if (C.ext[k] == C.pair1) jp = k;
  }
  const long total = ntot * inner;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long t = e / inner;
    const long r = e % inner;
    int co[3];
    for (int k = C.next - 1; k >= 0; --k) {
      co[k] = t % ed.d[k];
      t /= ed.d[k];
    }
    const int x = co[ip];
    co[ip] = co[jp];
    co[jp] = x;
    dst[e] = src[tuple_index(C, ed.d, co) * inner + r];
  }
}

// Split-K Gram product over a tensor viewed as [pre][Ns][post]:
//   part[z][x][y] = sum_{k in chunk z} A(x, k) B(y, k),  k = (p, q) over pre x post,
//   A(x, (p, q)) = A[(p * Ns + x) * post + q].
// Output tile 32 x 32 per block: lanes over y, rows x dealt to the eight warps and skipped
// beyond Ns (Ns is often 4 to 20: every FP64 instruction of a warp costs its sub-partition
// 64 clocks, idle lanes or not), K staged in chunks of 32 through shared memory.
constexpr int kGS = 32, kGK = 32;
__global__ void __launch_bounds__(256)
k_gram(const double* __restrict__ A, const double* __restrict__ B, long Ns, unsigned post,
       unsigned K, unsigned chunk, double* __restrict__ part) {
  __shared__ double sa[kGK][kGS + 1], sb[kGK][kGS + 1];
  const long x0 = (long)blockIdx.y * kGS, y0 = (long)blockIdx.x * kGS;
  const unsigned kbeg = blockIdx.z * chunk;
  const unsigned kend = min(K, kbeg + chunk);
  const bool xfast = post == 1u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nx = (int)min((long)kGS, Ns - x0), ny = (int)min((long)kGS, Ns - y0);
  const int nr = max(0, min(4, (nx - warp + 7) / 8));
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (unsigned k0 = kbeg; k0 < kend; k0 += kGK) {
#pragma unroll
    for (int u = 0; u < kGK * kGS / 256; ++u) {
      const int l = threadIdx.x + 256 * u;
      int kk, ii;
      if (xfast) { ii = l % kGS; kk = l / kGS; } else { kk = l % kGK; ii = l / kGK; }
      const unsigned gk = k0 + kk;
      double va = 0.0, vb = 0.0;
      if (gk < kend && (ii < nx || ii < ny)) {
        const unsigned p = gk / post, q = gk - p * post;
        const long base = (long)p * Ns * post + q;
        if (ii < nx) va = A[base + (x0 + ii) * post];
        if (ii < ny) vb = B[base + (y0 + ii) * post];
      }
      sa[kk][ii] = va;
      sb[kk][ii] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (r < nr) {
#pragma unroll 8
        for (int kk = 0; kk < kGK; ++kk) acc[r] = fma(sa[kk][warp + 8 * r], sb[kk][lane], acc[r]);
      }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (r < nr && lane < ny)
      part[((long)blockIdx.z * Ns + x0 + warp + 8 * r) * Ns + y0 + lane] = acc[r];
}

// Fixed-order sum of the split-K partials (a warp per element, lanes striding the partials,
// then a shuffle tree).  mode 0: out[x][y] = X; mode 1 (closed block): out[off + y][off + x] -=
// X; mode 2 (virtual block): out[off + x][off + y] += X.
__global__ void k_gram_finish(const double* __restrict__ part, int nsplit, long Ns, int mode,
                              double* __restrict__ out, long ld, long off) {
  const long total = Ns * Ns;
  const int lane = threadIdx.x & 31;
  const long nw = (long)gridDim.x * (blockDim.x >> 5);
  for (long e = blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5); e < total; e += nw) {
    double s = 0.0;
    for (int z = lane; z < nsplit; z += 32) s += part[(long)z * total + e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane != 0) continue;
    const long x = e / Ns, y = e % Ns;
    if (mode == 0) out[x * ld + y] = s;
    else if (mode == 1) out[(off + y) * ld + off + x] -= s;
    else out[(off + x) * ld + off + y] += s;
  }
}

// The same with one partial: a thread per element.
__global__ void k_gram_place(const double* __restrict__ X, long Ns, int mode,
                             double* __restrict__ out, long ld, long off) {
  const long total = Ns * Ns;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long x = e / Ns, y = e % Ns;
    if (mode == 0) out[x * ld + y] = X[e];
    else if (mode == 1) out[(off + y) * ld + off + x] -= X[e];
    else out[(off + x) * ld + off + y] += X[e];
  }
}

// Active block of d2: partial sums over (row, col) of D^pi[row][col] dF_act^pi/df_uw.
// Each thread takes its own (row, col) elements, evaluates every plan term once (as the
// forward evaluation does) and adds coeff * D * Gamma into its private column of
// acc[uw][thread] in shared memory at uw = (f index 0, f index 1); a fixed-order sum over
// the threads gives part[block][a^2].  split: the warps of a block share 32 elements and deal
// the plan terms (small class matrices).
__global__ void k_act_adj(const ActPlan* __restrict__ plans, int nplan, DevClass C, int a, int n,
                          RdmPtrs g, const double* __restrict__ Dm, int m, int split,
                          double* __restrict__ part) {
  extern __shared__ double acc[];   // [a^2][blockDim.x]
  const int a2 = a * a, nt = blockDim.x, tid = threadIdx.x;
  for (int q = 0; q < a2; ++q) acc[q * nt + tid] = 0.0;
  const long total = (long)m * m;
  const long A = ipow(a, C.nact);
  const int per = split ? 32 : nt;                 // elements of a block at a time
  const int t0 = split ? tid >> 5 : 0, ts = split ? nt >> 5 : 1;
  for (long e = (long)blockIdx.x * per + (split ? tid & 31 : tid); e < total;
       e += (long)gridDim.x * per) {
    const double D0 = Dm[e], D1 = Dm[total + e];
    if (D0 == 0.0 && D1 == 0.0) continue;
    const int row = e / m, col = e % m;
    int vals[24];
    const int M = row % n, N = col % n;
    long ab = row / n, ak = col / n;
    const int fb = ab / A, fk = ak / A;
    ab %= A;
    ak %= A;
    for (int k = C.nact - 1; k >= 0; --k) {
      vals[kRefBra + k] = ab % a;
      ab /= a;
      vals[kRefKet + k] = ak % a;
      ak /= a;
    }
    for (int t = t0; t < nplan; t += ts) {
      const ActPlan& P = plans[t];
      if (!P.has_f || P.fb != fb || P.fk != fk) continue;
      const double Dv = P.pi == 0 ? D0 : D1;
      if (Dv == 0.0) continue;
      bool ok = true;
      for (int q = 0; q < P.neq; ++q)
        if (vals[P.eq[q][0]] != vals[P.eq[q][1]]) ok = false;
      if (!ok) continue;
      const int nl = P.nloop;
      const int niter = nl == 0 ? 1 : (nl == 1 ? a : a * a);
      const double cd = P.coeff * Dv;
      for (int it = 0; it < niter; ++it) {
        if (nl >= 1) vals[kRefLoop] = it % a;
        if (nl >= 2) vals[kRefLoop + 1] = it / a;
        const double x = rdm_at(g.p, P.rank, n, a, M, N, vals, P.idx);
        const int uw = vals[P.fidx[0]] * a + vals[P.fidx[1]];
        acc[uw * nt + tid] += cd * x;
      }
    }
  }
  __syncthreads();
  for (int q = tid >> 5; q < a2; q += nt >> 5) {
    double t = 0.0;
    for (int j = tid & 31; j < nt; j += 32) t += acc[q * nt + j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((tid & 31) == 0) part[(long)blockIdx.x * a2 + q] = t;
  }
}

// d2[c + u][c + w] += sum_blocks part[b][uw] - sum_L NL[L] Gamma1[L][L][u][w]
__global__ void k_act_finish(const double* __restrict__ part, int nblk, int a, int c, int nmo,
                             const double* __restrict__ NL, const double* __restrict__ g1, int n,
                             double* __restrict__ d2) {
  const int a2 = a * a;
  for (int uw = threadIdx.x >> 5; uw < a2; uw += blockDim.x >> 5) {
    double s = 0.0;
    for (int b = threadIdx.x & 31; b < nblk; b += 32) s += part[(long)b * a2 + uw];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) != 0) continue;
    for (int L = 0; L < n; ++L) s -= NL[L] * g1[((long)L * n + L) * a2 + uw];
    d2[(long)(c + uw / a) * nmo + c + uw % a] += s;
  }
}

// Source multipliers W = r_L' sum_L r_L T_L + Lam_L' in the layout of the sources V,
// W[fam][t][act][M][L'], from T, Lam [t][L][(fam, act, M)].
__global__ void k_wsrc(const double* __restrict__ T, const double* __restrict__ Lam,
                       const double* __restrict__ R, int P, int n, long m, long ntot, int nfam,
                       double* __restrict__ W) {
  const long total = ntot * m, per = m / nfam;    // per = A n rows of a family
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long row = e % m, t = e / m;
    double acc = 0.0;
    for (int L = 0; L < n; ++L) acc += R[L * n + P] * T[(t * n + L) * m + row];
    double* w = W + (((row / per) * ntot + t) * per + row % per) * n;
    for (int Lp = 0; Lp < n; ++Lp) w[Lp] = R[Lp * n + P] * acc + Lam[(t * n + Lp) * m + row];
  }
}

__device__ __forceinline__ void flush_add(double* p, double v) {
  if (p != nullptr && v != 0.0) atomicAdd(p, v);
}

// Target of an integral of a source term: element of d1 (kind 0), of the adjoint (pq|rt) block
// (kind 1) or of the adjoint of a pre-summed block (kind 2).
struct AdjTarget {
  double* base;
  long s0, s1, s2;             // strides of the first three indices (the last is contiguous)
  int o0, o1;                  // offsets of the first two (kind 0)
};
__device__ __forceinline__ AdjTarget adj_target(int kind, int cb, const int8_t* sp, const Dims& d,
                                                double* d1, const EriBlocks& G,
                                                const PresumBlocks& GP) {
  const int dimsp[4] = {d.c, d.a, d.v, 1};
  const int offsp[3] = {0, d.c, d.c + d.a};
  if (kind == 0) return {d1, 0, 0, d.nmo(), offsp[sp[0]], offsp[sp[1]]};
  const long s2 = dimsp[sp[3]], s1 = s2 * dimsp[sp[2]], s0 = s1 * dimsp[sp[1]];
  double* b = const_cast<double*>(
      kind == 1 ? G.p[((sp[0] * 3 + sp[1]) * 3 + sp[2]) * 3 + sp[3]] : GP.p[cb]);
  return {b, s0, s1, s2, 0, 0};
}
__device__ __forceinline__ double* adj_element(const AdjTarget& t, int kind, const int* vals,
                                               const int8_t* idx) {
  if (kind == 0) return t.base + (t.o0 + vals[idx[0]]) * t.s2 + t.o1 + vals[idx[1]];
  return t.base + vals[idx[0]] * t.s0 + vals[idx[1]] * t.s1 + vals[idx[2]] * t.s2 + vals[idx[3]];
}

// Adjoint of the sources that the plan interpreter forms: for every (fam, ext, act) and the
// n^2 multipliers W[M][L'], each plan term adds coeff * sum_(M,L') W Gamma[M][L'][off] to its
// integral's target, with one atomic add per run of equal targets.  NS = n holds the
// multipliers in registers; NS = 0 reads them (any n).  TG warps share 32 elements and deal
// the plan terms (TG = 1: one thread an element).
template <int NS, int TG>
__global__ void __launch_bounds__(256)
k_src_adj(const SrcPlan* __restrict__ plans, int nplan, DevClass C, Dims d, RdmPtrs g,
          const double* __restrict__ W, long total2, double* __restrict__ d1, EriBlocks G,
          PresumBlocks GP) {
  const int n = NS > 0 ? NS : d.n, a = d.a;
  const int dimsp[4] = {d.c, d.a, d.v, 1};
  constexpr int per = 256 / TG;
  for (long e = (long)blockIdx.x * per + threadIdx.x % per; e < total2;
       e += (long)gridDim.x * per) {
    long r = e;
    int vals[24];
    vals[kRefZero] = 0;
    for (int k = C.nact - 1; k >= 0; --k) {
      vals[kRefBra + C.act[k]] = r % a;
      r /= a;
    }
    for (int k = C.next - 1; k >= 0; --k) {
      const int dm = dimsp[C.slot_space[C.ext[k]]];
      vals[kRefBra + C.ext[k]] = r % dm;
      r /= dm;
    }
    const int fam = (int)r;
    const double* wp = W + e * n * n;
    double wv[NS > 0 ? NS * NS : 1];
    if (NS > 0) {
#pragma unroll
      for (int q = 0; q < NS * NS; ++q) wv[q] = wp[q];
    }
    double* last = nullptr;
    double run = 0.0;
    for (int tp = threadIdx.x / per; tp < nplan; tp += TG) {
      const SrcPlan& P = plans[tp];
      if (P.fb != fam) continue;
      bool ok = true;
      for (int qq = 0; qq < P.neq; ++qq)
        if (vals[P.eq[qq][0]] != vals[P.eq[qq][1]]) ok = false;
      if (!ok) continue;
      long niter = 1;
      for (int j = 0; j < P.nloop; ++j) niter *= dimsp[P.loop_space[j]];
      const AdjTarget at = adj_target(P.kind, P.cb, P.ispace, d, d1, G, GP);
      const long stride = ipow(a, 2 * P.rank);
      for (long it = 0; it < niter; ++it) {
        long qi = it;
        for (int j = 0; j < P.nloop; ++j) {
          const int dm = dimsp[P.loop_space[j]];
          vals[kRefLoop + j] = qi % dm;
          qi /= dm;
        }
        double gs = 0.0;
        if (P.rank == 0) {
          for (int M = 0; M < n; ++M) gs += NS > 0 ? wv[M * n + M] : wp[M * n + M];
        } else {
          long off = 0;
          for (int j = 0; j < 2 * P.rank; ++j) off = off * a + vals[P.idx[j]];
          const double* gp = g.p[P.rank] + off;
          if (NS > 0) {
#pragma unroll
            for (int q = 0; q < NS * NS; ++q) gs = fma(wv[q], gp[q * stride], gs);
          } else {
            for (int q = 0; q < n * n; ++q) gs = fma(wp[q], gp[q * stride], gs);
          }
        }
        if (gs == 0.0) continue;
        double* tgt = adj_element(at, P.kind, vals, P.iidx);
        if (tgt != last) {
          flush_add(last, run);
          last = tgt;
          run = 0.0;
        }
        run += P.coeff * gs;
      }
    }
    flush_add(last, run);
  }
}

// Adjoint of k_src_x: the adjoint XA[row][k] of a source group's X, over the external tuples
// row0 .. row0 + nrow, times each integral term's coefficient, added to the term's target.
__global__ void k_src_x_adj(const SrcXTerm* __restrict__ xt, int nx, DevClass C, Dims d, int ns,
                            const double* __restrict__ XA, long row0, long nrow,
                            double* __restrict__ d1, EriBlocks G, PresumBlocks GP) {
  const int a = d.a;
  const int dimsp[4] = {d.c, d.a, d.v, 1};
  const long K = ipow(a, ns);
  const long total = nrow * K;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const double xa = XA[e];
    if (xa == 0.0) continue;
    int vals[32];
    vals[kRefZero] = 0;
    long q = e % K;
    for (int p = ns - 1; p >= 0; --p) {
      vals[kRefLoop + p] = (int)(q % a);
      q /= a;
    }
    long r = row0 + e / K;
    for (int k = C.next - 1; k >= 0; --k) {
      const int dm = dimsp[C.slot_space[C.ext[k]]];
      vals[kRefBra + C.ext[k]] = (int)(r % dm);
      r /= dm;
    }
    for (int t = 0; t < nx; ++t) {
      const SrcXTerm& T = xt[t];
      bool ok = true;
      for (int u = 0; u < T.neq; ++u)
        if (vals[T.eq[u][0]] != vals[T.eq[u][1]]) ok = false;
      if (!ok) continue;
      const AdjTarget at = adj_target(T.kind, T.cb, T.ispace, d, d1, G, GP);
      long niter = 1;
      for (int j = 0; j < T.nloop; ++j) niter *= dimsp[T.loop_space[j]];
      for (long it = 0; it < niter; ++it) {
        long w = it;
        for (int j = 0; j < T.nloop; ++j) {
          const int dm = dimsp[T.loop_space[j]];
          vals[kRefLoop + ns + j] = (int)(w % dm);
          w /= dm;
        }
        atomicAdd(adj_element(at, T.kind, vals, T.iidx), T.coeff * xa);
      }
    }
  }
}

__global__ void k_symmetrize(double* __restrict__ x, int nmo, long batch) {
  const long nn = (long)nmo * nmo;
  const long total = batch * nn;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long r = e % nn;
    const int i = r / nmo, j = r % nmo;
    if (i >= j) continue;
    double* m = x + (e - r);
    const double s = 0.5 * (m[(long)i * nmo + j] + m[(long)j * nmo + i]);
    m[(long)i * nmo + j] = s;
    m[(long)j * nmo + i] = s;
  }
}

}  // namespace

// X = sum over (pre, post) of A(x, .) B(y, .) for [pre][Ns][post] tensors, finished
// into `out` according to `mode` (see k_gram_finish).
int gram_product(const double* A, const double* B, long pre, long Ns, long post, int mode,
                 double* out, long ld, long off, double* part, long partmax, cudaStream_t s,
                 OzWork* oz) {
  if (pre * Ns * post == 0) return CASPT2_OK;
  const long K = pre * post;
  if (K >= (1L << 31) || Ns * Ns > partmax) return CASPT2_EINVAL;
  if (oz && oz->on) {
    // element (x, (p, q)) of a [pre][Ns][post] tensor: x * post + p * Ns * post + q
    const OzView va{A, post, 1, post, Ns * post}, vb{B, post, 1, post, Ns * post};
    CASPT2_CUDA_TRY(oz_matmul(*oz, va, vb, A == B, (int)Ns, (int)Ns, (int)K, 1.0, 0.0, part, Ns,
                              s));
    ++launch_counter();
    k_gram_place<<<launch_blocks(Ns * Ns), 256, 0, s>>>(part, Ns, mode, out, ld, off);
    CASPT2_CUDA_TRY(cudaGetLastError());
    return CASPT2_OK;
  }
  const long ntile = (Ns + kGS - 1) / kGS;
  const long tiles = ntile * ntile;
  // four blocks a SM, each with at least four chunks of K
  long nsplit = std::max<long>(1, (152L * 4 + tiles - 1) / tiles);
  nsplit = std::min(nsplit, std::max<long>(1, K / (4 * kGK)));
  nsplit = std::min(nsplit, partmax / (Ns * Ns));
  long chunk = (K + nsplit - 1) / nsplit;
  chunk = (chunk + kGK - 1) / kGK * kGK;
  nsplit = (K + chunk - 1) / chunk;
  dim3 grid((unsigned)ntile, (unsigned)ntile, (unsigned)nsplit);
  ++launch_counter();
  k_gram<<<grid, 256, 0, s>>>(A, B, Ns, (unsigned)post, (unsigned)K, (unsigned)chunk, part);
  ++launch_counter();
  if (nsplit == 1)
    k_gram_place<<<launch_blocks(Ns * Ns), 256, 0, s>>>(part, Ns, mode, out, ld, off);
  else
    k_gram_finish<<<launch_blocks(Ns * Ns * 32), 256, 0, s>>>(part, (int)nsplit, Ns, mode, out, ld,
                                                             off);
  CASPT2_CUDA_TRY(cudaGetLastError());
  return CASPT2_OK;
}

long class_dens_tall(const ClassWork& w, const Dims& d) {
  if (w.vsize == 0 || w.m == 0) return 0;
  return all_tuples(w) * d.n * w.m;
}

cudaError_t launch_symmetrize(double* x, int nmo, long batch, cudaStream_t s) {
  const long total = batch * (long)nmo * nmo;
  if (total == 0) return cudaSuccess;
  ++launch_counter();
  k_symmetrize<<<launch_blocks(total), 256, 0, s>>>(x, nmo, batch);
  return cudaGetLastError();
}

int class_tuple_amplitudes(ClassWork& w, DensWork& dw, const Dims& d, double shift,
                           const double* E0, const double* eps_cv, const double* R, int P,
                           OzWork* oz, cudaStream_t s) {
  const int m = w.m, n = d.n;
  if (w.vsize == 0 || m == 0) return CASPT2_OK;
  const DevClass& C = w.dc;
  const long ntot = all_tuples(w);
  const long tall = ntot * n * m;
  if (tall > dw.tall) return CASPT2_EINVAL;
  CASPT2_CUDA_TRY(cudaMemsetAsync(dw.T, 0, sizeof(double) * tall, s));
  CASPT2_CUDA_TRY(cudaMemsetAsync(dw.Lam, 0, sizeof(double) * tall, s));

  // ---- amplitudes and lambda of every sector, back-transformed to all tuples
  for (const SectorKeep& K : w.keep) {
    if (K.nk == 0 || K.ntup == 0) continue;
    const int nL = K.Lsel < 0 ? n : 1;
    const long ncol = K.ntup * nL;
    if ((long)K.nk * ncol > dw.secmax || (long)K.msec * ncol > dw.secmax) return CASPT2_EINVAL;
    double* amp = dw.sec;
    double* lam = dw.sec + dw.secmax;
    ++launch_counter();
    k_sector_amp<<<launch_blocks((long)K.nk * ncol), 256, 0, s>>>(
        K.Vt, K.omega, E0, eps_cv, R, P, C, w.ed, d.c, n, K.sec, K.Lsel, K.ntup, K.nk, shift, amp,
        lam);
    CASPT2_CUDA_TRY(cudaGetLastError());
    // rows = Y (msec x nk) times sector columns, for amp and lam together
    if (oz && oz->on) {
      const OzView vy{K.Y, K.nk, 1, K.nk, 0};                   // rows i, K = mu
      for (int q = 0; q < 2; ++q) {
        const OzView vs{dw.sec + q * dw.secmax, 1, ncol, K.nk, 0};   // rows col, K = mu
        CASPT2_CUDA_TRY(oz_matmul(*oz, vy, vs, false, K.msec, (int)ncol, K.nk, 1.0, 0.0,
                                  dw.tmp + q * dw.secmax, ncol, s));
      }
    } else {
      CASPT2_CUDA_TRY(dgemm(K.msec, (int)ncol, K.nk, 1.0, K.Y, K.nk, false, dw.sec, (int)ncol,
                            false, 0.0, dw.tmp, (int)ncol, s, 2, 0, dw.secmax, dw.secmax));
    }
    ++launch_counter();
    k_tuple_scatter<<<launch_blocks((long)K.msec * ncol), 256, 0, s>>>(
        dw.tmp, dw.tmp + dw.secmax, C, w.ed, n, m, K.sec, K.Lsel, K.ntup, K.msec, dw.T, dw.Lam);
    CASPT2_CUDA_TRY(cudaGetLastError());
  }
  return CASPT2_OK;
}

int class_densities(ClassWork& w, DensWork& dw, SectorWork& sw, const Dims& d, int scheme,
                    double shift, RdmPtrs rdm, const double* E0, const double* eps_cv,
                    const double* R, int P, const double* NL, const EriBlocks& G,
                    const PresumBlocks& GP, double* d1, double* d2, OzWork* oz, cudaStream_t s) {
  (void)scheme;
  const int m = w.m, n = d.n, a = d.a, nmo = d.nmo();
  if (w.vsize == 0 || m == 0) return CASPT2_OK;
  const DevClass& C = w.dc;
  const long ntot = all_tuples(w);
  const long tall = ntot * n * m;
  if (a * a > 256) return CASPT2_EINVAL;
  {
    const int st = class_tuple_amplitudes(w, dw, d, shift, E0, eps_cv, R, P, oz, s);
    if (st != CASPT2_OK) return st;
  }
  const bool pair = C.pair0 >= 0;
  const long mm = (long)m * m;
  // ---- overlap applied to T: U1 = S^id T, U2 = S^sw T (rows of T are (tuple, L))
  if (oz && oz->on) {
    const OzView vt{dw.T, m, 1, m, 0}, vs1{w.Sact, m, 1, m, 0}, vs2{w.Sact + mm, m, 1, m, 0};
    CASPT2_CUDA_TRY(oz_matmul(*oz, vt, vs1, false, (int)(ntot * n), m, m, 1.0, 0.0, dw.U1, m, s));
    if (pair)
      CASPT2_CUDA_TRY(oz_matmul(*oz, vt, vs2, false, (int)(ntot * n), m, m, 1.0, 0.0, dw.U2, m, s));
  } else {
    CASPT2_CUDA_TRY(dgemm((int)(ntot * n), m, m, 1.0, dw.T, m, false, w.Sact, m, true, 0.0, dw.U1,
                          m, s));
    if (pair)
      CASPT2_CUDA_TRY(dgemm((int)(ntot * n), m, m, 1.0, dw.T, m, false, w.Sact + mm, m, true, 0.0,
                            dw.U2, m, s));
  }
  // ---- closed and virtual blocks: one external slot moves
  auto slot_blocks = [&](const double* Lm, const double* U) -> int {
    long pre = 1;
    for (int k = 0; k < C.next; ++k) {
      const long Ns = w.ed.d[k];
      long post = (long)n * m;
      for (int k2 = k + 1; k2 < C.next; ++k2) post *= w.ed.d[k2];
      const int sp = C.slot_space[C.ext[k]];
      const int st = gram_product(Lm, U, pre, Ns, post, sp == SP_C ? 1 : 2, d2, nmo,
                                  space_off(d, sp), dw.part, dw.partmax, s, oz);
      if (st != CASPT2_OK) return st;
      pre *= Ns;
    }
    return CASPT2_OK;
  };
  int st = slot_blocks(dw.Lam, dw.U1);
  if (st != CASPT2_OK) return st;
  if (pair) {
    ++launch_counter();
    k_swap_tuples<<<launch_blocks(tall), 256, 0, s>>>(dw.Lam, C, w.ed, ntot, (long)n * m, dw.Tsw);
    CASPT2_CUDA_TRY(cudaGetLastError());
    st = slot_blocks(dw.Tsw, dw.U2);
    if (st != CASPT2_OK) return st;
  }
  // ---- active block: D^pi = sum_(tuple, L) lambda x T^pi, contracted with dF_act/df
  st = gram_product(dw.Lam, dw.T, ntot * n, m, 1, 0, dw.Dm, m, 0, dw.part, dw.partmax, s, oz);
  if (st != CASPT2_OK) return st;
  if (pair) {
    ++launch_counter();
    k_swap_tuples<<<launch_blocks(tall), 256, 0, s>>>(dw.T, C, w.ed, ntot, (long)n * m, dw.Tsw);
    CASPT2_CUDA_TRY(cudaGetLastError());
    st = gram_product(dw.Lam, dw.Tsw, ntot * n, m, 1, 0, dw.Dm + mm, m, 0, dw.part, dw.partmax,
                      s, oz);
    if (st != CASPT2_OK) return st;
  } else {
    CASPT2_CUDA_TRY(cudaMemsetAsync(dw.Dm + mm, 0, sizeof(double) * mm, s));
  }
  if (a > 0) {
    const int a2 = a * a;
    // per-thread accumulator columns: at most 96 KB of shared memory per block
    const int nt = std::max(32, std::min(256, (int)(kActAdjSmem / (8L * a2)) / 32 * 32));
    const size_t smem = 8ull * a2 * nt;
    if (smem > (size_t)kActAdjSmem) return CASPT2_EINVAL;
    // terms dealt to the warps while a thread an element leaves the chip empty
    const int split = mm <= 152L * 4 * nt;
    const long nblk = std::max<long>(1, std::min<long>(152L * 4, split ? (mm + 31) / 32
                                                                       : (mm + nt - 1) / nt));
    if (nblk * a2 > dw.partmax) return CASPT2_EINVAL;
    CASPT2_CUDA_TRY(cudaFuncSetAttribute(k_act_adj, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kActAdjSmem));
    ++launch_counter();
    k_act_adj<<<(unsigned)nblk, nt, smem, s>>>(w.dF, w.nF, C, a, n, rdm, dw.Dm, m, split,
                                                dw.part);
    ++launch_counter();
    k_act_finish<<<1, 256, 0, s>>>(dw.part, (int)nblk, a, d.c, nmo, NL, rdm.p[1], n, d2);
    CASPT2_CUDA_TRY(cudaGetLastError());
  }
  // ---- sources: d1 and the adjoint integral blocks
  double* W = dw.U1;                 // [fam][tuple][act][M][L'], vsize doubles
  ++launch_counter();
  k_wsrc<<<launch_blocks(ntot * m), 256, 0, s>>>(dw.T, dw.Lam, R, P, n, m, ntot, C.nfam, W);
  CASPT2_CUDA_TRY(cudaGetLastError());
  if (w.nVs > 0) {
    const long total2 = w.vsize / ((long)n * n);
    const bool deal = total2 <= 152L * 4 * 256 && w.nVs > 1;
    auto run = [&](auto ns) {
      constexpr int NS = decltype(ns)::value;
      ++launch_counter();
      if (deal)
        k_src_adj<NS, 8><<<launch_blocks(total2, 32), 256, 0, s>>>(w.dVs, w.nVs, C, d, rdm, W,
                                                                   total2, d1, G, GP);
      else
        k_src_adj<NS, 1><<<launch_blocks(total2), 256, 0, s>>>(w.dVs, w.nVs, C, d, rdm, W, total2,
                                                               d1, G, GP);
    };
    if (n == 1) run(std::integral_constant<int, 1>());
    else if (n == 2) run(std::integral_constant<int, 2>());
    else if (n == 3) run(std::integral_constant<int, 3>());
    else if (n == 4) run(std::integral_constant<int, 4>());
    else run(std::integral_constant<int, 0>());
    CASPT2_CUDA_TRY(cudaGetLastError());
  }
  // the terms of the GEMM groups: the adjoint of V += X G is XA = W G^T, added to the targets
  // of X's integral terms (all of classes F and G: 17 of the 42 ms that one thread per source
  // element and term took at c20 a8 v200 n3)
  const long ncol = w.A * n * n;
  for (size_t gi = 0; gi < w.hG.size(); ++gi) {
    const SrcGemmGroup& Gr = w.hG[gi];
    const long K = ipow_host(a, Gr.g.ns);
    if (K * ncol > sw.srcGcap) return CASPT2_EINVAL;
    CASPT2_CUDA_TRY(launch_src_g(Gr.g, C, d, rdm, sw.srcG, s));
    const long chunk = std::min<long>(ntot, sw.srcXcap / K);
    if (chunk < 1) return CASPT2_EINVAL;
    for (long r0 = 0; r0 < ntot; r0 += chunk) {
      const long nr = std::min(chunk, ntot - r0);
      CASPT2_CUDA_TRY(dgemm((int)nr, (int)K, (int)ncol, 1.0, W + ((long)Gr.fb * ntot + r0) * ncol,
                            (int)ncol, false, sw.srcG, (int)ncol, true, 0.0, sw.srcX, (int)K, s));
      ++launch_counter();
      k_src_x_adj<<<launch_blocks(nr * K), 256, 0, s>>>(w.dX + w.gx_off[gi], (int)Gr.x.size(), C,
                                                        d, Gr.g.ns, sw.srcX, r0, nr, d1, G, GP);
      CASPT2_CUDA_TRY(cudaGetLastError());
    }
  }
  return CASPT2_OK;
}

namespace {
// out[fam][ext...][act...] = src[tuple][L][(fam, act..., N)] for one (L, N)
__global__ void k_gather_amp(const double* __restrict__ src, int nfam, long ntot, long A, int n,
                             int L, int N, double* __restrict__ out) {
  const long total = (long)nfam * ntot * A;
  const long m = (long)nfam * A * n;
  for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < total;
       o += (long)gridDim.x * blockDim.x) {
    const long act = o % A;
    const long t = (o / A) % ntot;
    const long fam = o / (A * ntot);
    out[o] = src[(t * n + L) * m + (fam * A + act) * n + N];
  }
}
}  // namespace

cudaError_t gather_amplitudes(const ClassWork& w, const Dims& d, const double* src, int L, int N,
                              double* out, cudaStream_t s) {
  const long total = (long)w.dc.nfam * all_tuples(w) * w.A;
  if (total == 0) return cudaSuccess;
  ++launch_counter();
  k_gather_amp<<<launch_blocks(total), 256, 0, s>>>(src, w.dc.nfam, all_tuples(w), w.A, d.n, L, N,
                                                    out);
  return cudaGetLastError();
}

}  // namespace caspt2
