// Device pieces of the symmetric tridiagonal eigenproblem shared by the one-block sector
// solver and the large-matrix path: Sturm counts, eigenvalues, inverse iteration.
#pragma once
#include "common.cuh"

namespace caspt2 {

// Where only the eigenvectors at or above a cut wmin are returned, those of the eigenvalues
// down to this bound are formed and orthogonalised with them: vectors from inverse iteration
// overlap by about eps ||T|| / gap, so a kept vector would carry 1e-9 of a dropped one a gap
// of 1e-6 below it.  What lies below 1e-4 of the cut has an overlap norm smaller by as much;
// what lies within the rounding of zero is the null space, which enters nothing.
__host__ __device__ inline double eig_guard(double wmin, double tnorm) {
  const double g = fmax(1e-4 * wmin, 1e-14 * tnorm);
  return g < wmin ? g : wmin;
}

// Bracket width at which an eigenvalue is taken (times ||T||, in the large-matrix path times
// max(1, ||T||)): half an FP64 rounding,
// so that the search adds nothing to the rounding of T.  The overlap's small eigenvalues
// normalise the range basis, s^(-1/2): at s = 1e-6 one rounding of ||T|| = 10 is 2e-9 of s.
constexpr double kEigTol = 1.1e-16;

__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ unsigned long long abits(double v) {   // |v| as an ordered integer
  return (unsigned long long)dbits(v) & 0x7FFFFFFFFFFFFFFFull;
}

// Last principal minor p_m(x) = det(T - x) and the number of eigenvalues of T below x, from
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (p_{-1} = 1): three FP64 operations per step
// and no division.  The count is the number of sign changes; signs, exact zeros (which take
// the sign opposite to their predecessor) and the range check are integer operations on the
// bit patterns.  The pair (p_i, p_{i-1}) is rescaled by 2^(-+500) when |p_i| leaves
// [2^-600, 2^600], checked every 4 steps (|p| grows by at most (2||T|| + ||T||^2) per step,
// far inside the FP64 range): p_m = val 2^(500 ex).
__device__ __forceinline__ int sturm_value(const double* __restrict__ d,
                                           const double* __restrict__ e2, int m, double x,
                                           double& val, int& ex) {
  double pm = 1.0, pc = d[0] - x;
  ex = 0;
  if ((dbits(pc) << 1) == 0) pc = -1e-300;
  int cnt = (int)((unsigned long long)dbits(pc) >> 63);
  for (int i = 1; i < m; ++i) {
    double pn = fma(d[i] - x, pc, -e2[i - 1] * pm);
    const long long bn = dbits(pn), bc = dbits(pc);
    if ((bn << 1) == 0) pn = bc < 0 ? 1e-300 : -1e-300;
    cnt += (int)((unsigned long long)(dbits(pn) ^ bc) >> 63);
    pm = pc;
    pc = pn;
    if ((i & 3) == 0) {
      const int xp = (int)((dbits(pc) >> 52) & 0x7FF);
      const int xm = (int)((dbits(pm) >> 52) & 0x7FF);
      if (xp > 1023 + 600) { pc *= 0x1p-500; pm *= 0x1p-500; ++ex; }
      else if (xp < 1023 - 600 && xm < 1023 - 600) { pc *= 0x1p500; pm *= 0x1p500; --ex; }
    }
  }
  val = pc;
  return cnt;
}

// Sturm count in single precision by the ratio recurrence q_i = d_i - x - e_(i-1)^2 / q_(i-1)
// (q raised to -pivmin where it vanishes): the count is exact for a tridiagonal matrix whose
// elements carry relative errors of a few float roundings, so it brackets every eigenvalue
// to within a few 2^-24 tnorm.
__device__ __forceinline__ int sturm_f32(const float* __restrict__ d,
                                         const float* __restrict__ e2, int m, float x,
                                         float pivmin) {
  float q = d[0] - x;
  if (fabsf(q) < pivmin) q = -pivmin;
  int cnt = q < 0.f ? 1 : 0;
  for (int i = 1; i < m; ++i) {
    q = (d[i] - x) - __fdividef(e2[i - 1], q);
    if (fabsf(q) < pivmin) q = -pivmin;
    cnt += q < 0.f ? 1 : 0;
  }
  return cnt;
}

// Width of the single-precision phase's brackets: 64 float roundings of the norm.
__device__ __forceinline__ double f32_gap(double glo, double ghi) {
  return 64.0 * 0x1p-24 * fmax(fabs(glo), fabs(ghi));
}
__device__ __forceinline__ bool f32_usable(double glo, double ghi) {
  const double span = fmax(fabs(glo), fabs(ghi));
  return span > 1e-20 && span < 1e18 && ghi - glo > 4.0 * f32_gap(glo, ghi);
}

// Single-precision bracket [flo, fhi] of eigenvalue j by octasection: the eight lanes of an
// aligned group count at the seven interior eighth points (three bits a pass).  The float
// units run 64 times the FP64 rate.  Every lane of the group calls it with the same j.
__device__ __forceinline__ void bisect_f32(const float* __restrict__ df,
                                           const float* __restrict__ ef, int m, int j, double glo,
                                           double ghi, float& flo, float& fhi) {
  flo = (float)glo;
  fhi = (float)ghi;
  if (!f32_usable(glo, ghi)) return;
  const unsigned sh = threadIdx.x & 24;
  const unsigned grp = 0xFFu << sh;
  const int q = threadIdx.x & 7;
  const double gap = f32_gap(glo, ghi);
  const float pivmin = (float)fmax(1e-30, 0x1p-24 * 1e-8 * fmax(fabs(glo), fabs(ghi)));
  for (int it = 0; it < 40; ++it) {
    if ((double)fhi - (double)flo <= gap) break;
    const float h = 0.125f * (fhi - flo);
    const float x = flo + h * (float)(q + 1);
    const bool above = q < 7 && x > flo && x < fhi && sturm_f32(df, ef, m, x, pivmin) > j;
    const unsigned b = (__ballot_sync(grp, above) >> sh) & 0x7Fu;
    const int first = b ? (__ffs(b) - 1) : 7;
    const float nhi = first < 7 ? flo + h * (float)(first + 1) : fhi;
    const float nlo = first > 0 ? flo + h * (float)first : flo;
    if (!(nhi < fhi || nlo > flo)) break;
    flo = nlo;
    fhi = nhi;
  }
}

// Eigenvalue j (ascending) of T to an absolute width tol, from its single-precision bracket.
// The bracket is widened by its uncertainty and both ends are checked with FP64 counts (an
// end that fails becomes the other end).  While it holds more than one eigenvalue it is
// halved; once it holds one, det(T - x) changes sign in it and the points come from the
// secant through the ends (Illinois: the kept end's value is halved when it is kept twice; a
// halving step whenever four steps did not shrink the bracket eightfold), the side always
// from the count.  About 9 evaluations of 3 m FP64 operations in place of the 35 bits of a
// bisection.  An eigenvalue that is known to lie below wmin is not refined further.
__device__ __forceinline__ double eigenvalue_f64(const double* __restrict__ d,
                                                 const double* __restrict__ e2, int m, int j,
                                                 double glo, double ghi, double flo, double fhi,
                                                 double tol, double wmin) {
  double lo = glo, hi = ghi, vlo = 0.0, vhi = 0.0;
  int cl = 0, ch = m, xlo = 0, xhi = 0;          // counts and exponents at the ends
  bool klo = false, khi = false;                 // values known
  int kept = 0, sec = 0;                         // > 0: lo kept that often, < 0: hi
  double wide = 0.0;
  const bool f32 = f32_usable(glo, ghi);
  const double gap = f32_gap(glo, ghi);
  int todo = f32 ? 2 : 0;
  for (int it = 0; it < 200; ++it) {
    double x;
    if (todo > 0) {
      x = todo == 2 ? flo - gap : fhi + gap;
      --todo;
      if (!(x > lo && x < hi)) continue;
    } else {
      // least distance of a point from the ends: a rounding of theirs where tol is below it
      const double ulp = 2.3e-16 * fmax(fabs(lo), fabs(hi)), step = fmax(0.75 * tol, ulp);
      if (hi - lo <= fmax(tol, ulp) || hi < wmin) break;
      x = 0.5 * (lo + hi);
      if (klo && khi && ch - cl == 1 && it < 60) {
        if ((sec & 3) == 0) {
          if (sec > 0 && hi - lo > 0.125 * wide) sec = -1;     // this step halves
          wide = hi - lo;
        }
        if (sec >= 0) {
          // vlo / (vlo - vhi); the ends' exponents may differ by a rescaling step
          double a = vlo, b = vhi;
          if (xlo > xhi) { a *= 0x1p250; b *= 0x1p-250; }
          else if (xlo < xhi) { a *= 0x1p-250; b *= 0x1p250; }
          const double t = abs(xlo - xhi) <= 1 ? a / (a - b) : (xlo > xhi ? 1.0 : 0.0);
          x = fma(t, hi - lo, lo);
          x = fmin(fmax(x, lo + step), hi - step);
          if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
        }
        ++sec;
      }
      if (!(x > lo && x < hi)) break;
    }
    double v;
    int ex;
    const int c = sturm_value(d, e2, m, x, v, ex);
    if (c > j) {
      hi = x; ch = c; vhi = v; xhi = ex; khi = true;
      kept = kept > 0 ? kept + 1 : 1;
      if (kept > 1) vlo *= 0.5;
    } else {
      lo = x; cl = c; vlo = v; xlo = ex; klo = true;
      kept = kept < 0 ? kept - 1 : -1;
      if (kept < -1) vhi *= 0.5;
    }
  }
  return 0.5 * (lo + hi);
}

// The same by an aligned group of eight lanes, for matrices whose eigenvalues leave the FP64
// units of other sub-partitions idle: every pass evaluates seven points at the latency of
// one.  While the bracket holds several eigenvalues they are its eighth points; once it
// holds one they lie around the secant point, at the least step and at the two geometric means
// between that and the width, with the midpoint: about three passes after the isolation.
// Every lane of the group calls it with the same j; the result is the group's.
__device__ __forceinline__ double eigenvalue_f64_group(const double* __restrict__ d,
                                                       const double* __restrict__ e2, int m,
                                                       int j, double glo, double ghi, double flo,
                                                       double fhi, double tol, double wmin) {
  const unsigned grp = 0xFFu << (threadIdx.x & 24);
  const int q = threadIdx.x & 7;
  double lo = glo, hi = ghi, vlo = 0.0, vhi = 0.0;
  int cl = 0, ch = m, xlo = 0, xhi = 0;
  bool klo = false, khi = false;
  const bool f32 = f32_usable(glo, ghi);
  const double gap = f32_gap(glo, ghi);
  for (int it = f32 ? -1 : 0; it < 60; ++it) {
    double x;
    bool use;
    if (it < 0) {                                // the single-precision bracket, widened
      x = q == 0 ? flo - gap : fhi + gap;
      use = q < 2;
    } else {
      const double ulp = 2.3e-16 * fmax(fabs(lo), fabs(hi)), step = fmax(0.75 * tol, ulp);
      const double width = hi - lo;
      if (width <= fmax(tol, ulp) || hi < wmin) break;
      if (klo && khi && ch - cl == 1 && it < 40) {
        double a = vlo, b = vhi;                 // exponents may differ by a rescaling step
        if (xlo > xhi) { a *= 0x1p250; b *= 0x1p-250; }
        else if (xlo < xhi) { a *= 0x1p-250; b *= 0x1p250; }
        const double t = abs(xlo - xhi) <= 1 ? a / (a - b) : (xlo > xhi ? 1.0 : 0.0);
        const double xs = fma(t, width, lo);
        const float l0 = log2f((float)step), l1 = log2f((float)width);
        const int lev = q >> 1;                  // 0, 1, 2 (two lanes each), 3: midpoint
        const double off = lev == 0 ? step
                                    : (double)exp2f(l0 + (l1 - l0) * (float)lev * (1.f / 3.f));
        x = lev == 3 ? lo + 0.5 * width : (q & 1 ? xs + off : xs - off);
      } else {
        x = lo + 0.125 * width * (q + 1);
      }
      use = q < 7;
    }
    use = use && x > lo && x < hi;
    double v = 0.0;
    int ex = 0, c = 0;
    if (use) c = sturm_value(d, e2, m, x, v, ex);
    __syncwarp(grp);
    bool moved = false;
#pragma unroll
    for (int r = 0; r < 7; ++r) {
      const double xr = __shfl_sync(grp, x, r, 8), vr = __shfl_sync(grp, v, r, 8);
      const int cr = __shfl_sync(grp, c, r, 8), er = __shfl_sync(grp, ex, r, 8);
      const bool ur = __shfl_sync(grp, use ? 1 : 0, r, 8) != 0;
      if (!ur) continue;
      if (cr > j) {
        if (xr < hi) { hi = xr; ch = cr; vhi = vr; xhi = er; khi = true; moved = true; }
      } else if (xr > lo) {
        lo = xr; cl = cr; vlo = vr; xlo = er; klo = true; moved = true;
      }
    }
    if (!moved && it >= 0) break;                // no representable point left inside
  }
  return 0.5 * (lo + hi);
}

__device__ __forceinline__ double hash_unit(unsigned a, unsigned b) {
  unsigned h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return (double)(h & 0xFFFFFF) / 16777216.0 + 0.5;   // in [0.5, 1.5)
}

// Shift of the inverse iteration for eigenvalue j of the nc ascending ones: equal eigenvalues are
// offset by 64 roundings of the norm.  At the eigenvalue itself the factorisation singles out one
// direction of their space, the same for all of them, and the Gram-Schmidt that follows would be
// left with rounding; at the offset every direction grows alike and the starts stay independent.
__device__ __forceinline__ double inverse_shift(const double* __restrict__ w, int nc, int j,
                                                double tnorm) {
  const double near = 1e-12 * tnorm, x = w[j];
  const bool close = (j > 0 && x - w[j - 1] <= near) || (j + 1 < nc && w[j + 1] - x <= near);
  return close ? x + 64 * 2.2e-16 * tnorm : x;
}

// Unit eigenvector j of nc for the shift lam by three inverse iterations from a fixed
// start vector, on the pivoted factorisation T - lam = P L U (U with two superdiagonals; a
// pivot below eps ||T|| is raised to it).  One thread a vector; scr holds [i][j] arrays (4 m nc
// doubles and m nc bytes), so that threads access consecutive addresses; Z[i * nc + j].  The
// rows of U are stored divided by their pivots, which leaves one FMA a row on the dependent
// chain of the back substitution; both passes load eight rows ahead of the chain.
__device__ __forceinline__ void inverse_iteration(const double* __restrict__ d,
                                                  const double* __restrict__ e, int m, double lam,
                                                  double tnorm, int nc, int j,
                                                  double* __restrict__ scr,
                                                  double* __restrict__ Z) {
  const long mn = (long)m * nc;
  double *rp = scr + j, *u1 = rp + mn, *u2 = u1 + mn, *lm = u2 + mn;
  unsigned char* pv = reinterpret_cast<unsigned char*>(scr + 4 * mn) + j;
  Z += j;
  const double tiny = 2.2e-16 * (tnorm > 0 ? tnorm : 1.0);
  const unsigned long long tbits = abits(tiny);
  auto raised = [&](double piv) { return abits(piv) < tbits ? copysign(tiny, piv) : piv; };
  // the current row (a, b) is carried in registers; rows are final once passed
  double a = d[0] - lam, b = m > 1 ? e[0] : 0.0;
  for (int i = 0; i < m - 1; ++i) {
    const double c = e[i];                       // subdiagonal element of row i + 1
    const double an = d[i + 1] - lam, bn = (i + 1 < m - 1) ? e[i + 1] : 0.0;
    const bool keep = abits(a) >= abits(c);
    const double r = recip(raised(keep ? a : c));
    const double l = (keep ? c : a) * r;
    const double s1 = keep ? b : an;             // U's first superdiagonal element
    rp[(long)i * nc] = r;
    u1[(long)i * nc] = s1 * r;
    u2[(long)i * nc] = keep ? 0.0 : bn * r;
    lm[(long)i * nc] = l;
    pv[(long)i * nc] = keep ? 0 : 1;
    a = fma(-l, s1, keep ? an : b);
    b = keep ? bn : -l * bn;
  }
  rp[(long)(m - 1) * nc] = recip(raised(a));
  u1[(long)(m - 1) * nc] = 0.0;
  u2[(long)(m - 1) * nc] = 0.0;
  constexpr int CH = 8;
  double nrm = 0.0;
  for (int iter = 0; iter < 3; ++iter) {
    // L^-1 with the row interchanges
    double cur = iter == 0 ? hash_unit(0, j) : Z[0];
    for (int i0 = 0; i0 < m - 1; i0 += CH) {
      const int cnt = min(CH, m - 1 - i0);
      double yv[CH], lv[CH];
      unsigned char pq[CH];
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (u < cnt) {
          const long o = (long)(i0 + u) * nc;
          yv[u] = iter == 0 ? hash_unit(i0 + u + 1, j) : Z[o + nc];
          lv[u] = lm[o];
          pq[u] = pv[o];
        }
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (u < cnt) {
          const double top = pq[u] ? yv[u] : cur, rest = pq[u] ? cur : yv[u];
          Z[(long)(i0 + u) * nc] = top;
          cur = fma(-lv[u], top, rest);
        }
    }
    Z[(long)(m - 1) * nc] = cur;
    // U^-1 (x1 = x_{i+1}, x2 = x_{i+2}); the norm of the last iterate on the way
    double x1 = 0.0, x2 = 0.0, n0 = 0.0, n1 = 0.0;
    for (int i0 = m - 1; i0 >= 0; i0 -= CH) {
      const int cnt = min(CH, i0 + 1);
      double zr[CH], c1[CH], c2[CH];
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (u < cnt) {
          const long o = (long)(i0 - u) * nc;
          zr[u] = Z[o] * rp[o];
          c1[u] = u1[o];
          c2[u] = u2[o];
        }
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (u < cnt) {
          const double x = fma(-c1[u], x1, fma(-c2[u], x2, zr[u]));
          Z[(long)(i0 - u) * nc] = x;
          if (iter == 2) {
            if (u & 1) n1 = fma(x, x, n1);
            else n0 = fma(x, x, n0);
          }
          x2 = x1;
          x1 = x;
        }
      // a chunk of eight rows grows by less than 1e130: rescale the partial solution when
      // its head passes 1e90
      if (abits(x1) > abits(1e90)) {
        const double f = 1.0 / fabs(x1);
        const int r0 = i0 - cnt + 1;
        for (int i = r0; i < m; ++i) Z[(long)i * nc] *= f;
        // rows above are not scaled: they hold L^-1 y, so their right-hand sides shrink too
        for (int i = 0; i < r0; ++i) Z[(long)i * nc] *= f;
        x1 *= f;
        x2 *= f;
        n0 = 0.0;
        n1 = 0.0;
        if (iter == 2)
          for (int i = r0; i < m; ++i) n0 = fma(Z[(long)i * nc], Z[(long)i * nc], n0);
      }
    }
    nrm = n0 + n1;
  }
  if (!(nrm < 1e290)) {                          // squares out of range: scale by the largest
    double big = 0.0;
    for (int i = 0; i < m; ++i) big = fmax(big, fabs(Z[(long)i * nc]));
    const double g = 1.0 / big;
    nrm = 0.0;
    for (int i = 0; i < m; ++i) {
      const double z = Z[(long)i * nc] * g;
      Z[(long)i * nc] = z;
      nrm = fma(z, z, nrm);
    }
  }
  const double f = 1.0 / sqrt(nrm);
  for (int i = 0; i < m; ++i) Z[(long)i * nc] *= f;
}

}  // namespace caspt2
