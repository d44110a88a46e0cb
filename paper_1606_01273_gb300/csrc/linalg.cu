// FP64 dense building blocks: tiled GEMMs, and the choice of the symmetric eigensolver.
#include <cooperative_groups.h>

#include "linalg.cuh"
#include "sector_block.cuh"

namespace cg = cooperative_groups;

namespace caspt2 {

// One tile of C = alpha op(A) op(B) + beta C: 32 x 32 outputs per block, lanes over the columns
// and rows dealt to the eight warps (warp w takes rows w, w + 8, ..), K in chunks of 16
// through shared memory with the next chunk's loads in flight.
//
// What bounds it: an SM's FP64 units take two lane operations a clock, so a tile's 1024 FMAs
// per k take 512 clocks against 512 bytes of operands: neither L2 nor shared memory is near
// its limit and the tile may be small.  What costs is FP64 work for padding and idle SMs.
// Rows beyond the edge are skipped by whole warps (M = 24 costs three quarters of M = 32; the
// dispatch transposes the product when that wastes fewer lanes), and a product with fewer
// tiles than the chip holds blocks splits K over a cluster of up to eight, whose partial
// tiles are summed through distributed shared memory in rank order.
constexpr int kGT = 32, kGK = 16;
struct GemmArgs {
  int M, N, K;
  double alpha, beta;
  const double* A; long ai, ak;      // A(i, k) = A[i ai + k ak]
  const double* B; long bk, bj;
  double* C; long ci, cj;
  long sA, sB, sC;                   // batch strides (blockIdx.y)
  unsigned akin, bkin;               // K in runs of akin (bkin) elements, the runs akout
  long akout, bkout;                 // (bkout) apart; a run as long as K: one run
  int tn, kc, split, sym;            // column tiles, K per block (multiple of kGK), cluster size
};

__global__ void __launch_bounds__(256) k_dgemm(GemmArgs g) {
  __shared__ double sa[2][kGK][kGT + 1], sb[2][kGK][kGT + 1];
  __shared__ double red[kGT][kGT + 1];
  const double* A = g.A + blockIdx.y * g.sA;
  const double* B = g.B + blockIdx.y * g.sB;
  double* C = g.C + blockIdx.y * g.sC;
  const int tile = blockIdx.x / g.split, rank = blockIdx.x % g.split;
  int by, bx;
  if (g.sym) {                       // symmetric result: upper-triangle tiles only
    int rem = tile;
    by = 0;
    while (rem >= g.tn - by) { rem -= g.tn - by; ++by; }
    bx = by + rem;
  } else {
    by = tile / g.tn;
    bx = tile % g.tn;
  }
  const int i0 = by * kGT, j0 = bx * kGT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kbeg = rank * g.kc, kend = min(g.K, kbeg + g.kc);
  const int nr = max(0, min(4, (g.M - i0 - warp + 7) / 8));      // rows of this warp
  // this thread's two elements of each operand chunk, along the operand's unit stride
  int ia[2], ka[2], jb[2], kb[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int l = threadIdx.x + 256 * u;
    if (g.ai == 1) { ia[u] = l % kGT; ka[u] = l / kGT; } else { ka[u] = l % kGK; ia[u] = l / kGK; }
    if (g.bj == 1) { jb[u] = l % kGT; kb[u] = l / kGT; } else { kb[u] = l % kGK; jb[u] = l / kGK; }
  }
  double va[2], vb[2];
  auto at = [](int k, long st, unsigned kin, long kout) {
    if ((unsigned)k < kin) return k * st;
    const unsigned p = (unsigned)k / kin;
    return p * kout + (k - p * kin) * st;
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int gi = i0 + ia[u], gk = k0 + ka[u];
      va[u] = (gi < g.M && gk < kend) ? A[gi * g.ai + at(gk, g.ak, g.akin, g.akout)] : 0.0;
      const int gj = j0 + jb[u], gq = k0 + kb[u];
      vb[u] = (gj < g.N && gq < kend) ? B[at(gq, g.bk, g.bkin, g.bkout) + gj * g.bj] : 0.0;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      sa[buf][ka[u]][ia[u]] = va[u];
      sb[buf][kb[u]][jb[u]] = vb[u];
    }
  };
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  if (kbeg < kend) {
    load(kbeg);
    store(0);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += kGK, buf ^= 1) {
    const bool more = k0 + kGK < kend;
    if (more) load(k0 + kGK);
    const double (*pa)[kGT + 1] = sa[buf], (*pb)[kGT + 1] = sb[buf];
    if (nr == 4) {
#pragma unroll 4
      for (int kk = 0; kk < kGK; ++kk) {
        const double b = pb[kk][lane];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fma(pa[kk][warp + 8 * r], b, acc[r]);
      }
    } else {
#pragma unroll
      for (int r = 0; r < 3; ++r)
        if (r < nr) {
#pragma unroll 4
          for (int kk = 0; kk < kGK; ++kk) acc[r] = fma(pa[kk][warp + 8 * r], pb[kk][lane], acc[r]);
        }
    }
    if (more) store(buf ^ 1);
    __syncthreads();
  }
  auto write = [&](int row, double x) {
    const int gi = i0 + row, gj = j0 + lane;
    if (gi >= g.M || gj >= g.N) return;
    double* c = C + gi * g.ci + gj * g.cj;
    *c = g.alpha * x + (g.beta == 0.0 ? 0.0 : g.beta * *c);
    if (g.sym && bx != by) {
      double* ct = C + gj * g.ci + gi * g.cj;
      *ct = g.alpha * x + (g.beta == 0.0 ? 0.0 : g.beta * *ct);
    }
  };
  if (g.split == 1) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (r < nr) write(warp + 8 * r, acc[r]);
    return;
  }
  cg::cluster_group cl = cg::this_cluster();
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (r < nr) red[warp + 8 * r][lane] = acc[r];
  cl.sync();
  // this rank finishes the rows equal to its rank modulo the cluster size
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = warp + 8 * r;
    if (r >= nr || row % g.split != rank) continue;
    double x = 0.0;
    for (int q = 0; q < g.split; ++q) x += *cl.map_shared_rank(&red[row][lane], q);
    write(row, x);
  }
  cl.sync();                         // the tiles stay readable until every rank is done
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

namespace {
// tiles: output tiles of one product; the rest of the grid and the launch.
cudaError_t launch_dgemm(GemmArgs g, long tiles, int batch, double flops, cudaStream_t s) {
  if (g.akin == 0) g.akin = 0xFFFFFFFFu;
  if (g.bkin == 0) g.bkin = 0xFFFFFFFFu;
  // K over a cluster while the blocks do not fill the chip (two a SM) and a block keeps at
  // least two chunks: 48 tiles of K = 1024 take 8.1 us a unit of K unsplit and 8.1 / 6 split
  int split = 1;
  while (split < 8 && tiles * batch * (split + 1) <= 2 * 152 && g.K >= 2 * kGK * (split + 1)) ++split;
  g.kc = (int)(((long)g.K + split - 1) / split + kGK - 1) / kGK * kGK;
  split = std::max(1, std::min(split, (g.K + g.kc - 1) / std::max(g.kc, 1)));
  g.split = split;
  ++launch_counter();
  const int slot = gemm_timer_begin(s);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * split), (unsigned)batch, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)split;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_dgemm, g);
  gemm_timer_end(slot, flops, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}
}  // namespace

cudaError_t dgemm(int M, int N, int K, double alpha, const double* A, int lda, bool ta,
                  const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                  cudaStream_t s, int batch, long sA, long sB, long sC) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  GemmArgs g{};
  g.K = K;
  g.alpha = alpha;
  g.beta = beta;
  g.C = C;
  // warp instructions per k: rows in eighths, columns in lanes of 32
  const long straight = (long)((M + 7) / 8) * ((N + 31) / 32);
  const long turned = (long)((N + 7) / 8) * ((M + 31) / 32);
  if (straight <= turned) {
    g.M = M; g.N = N;
    g.A = A; g.ai = ta ? 1 : lda; g.ak = ta ? lda : 1; g.sA = sA;
    g.B = B; g.bk = tb ? 1 : ldb; g.bj = tb ? ldb : 1; g.sB = sB;
    g.ci = ldc; g.cj = 1;
  } else {                           // C^T = op(B)^T op(A)^T
    g.M = N; g.N = M;
    g.A = B; g.ai = tb ? ldb : 1; g.ak = tb ? 1 : ldb; g.sA = sB;
    g.B = A; g.bk = ta ? lda : 1; g.bj = ta ? 1 : lda; g.sB = sA;
    g.ci = 1; g.cj = ldc;
  }
  g.sC = sC;
  g.tn = (g.N + kGT - 1) / kGT;
  const long tiles = (long)((g.M + kGT - 1) / kGT) * g.tn;
  return launch_dgemm(g, tiles, batch, 2.0 * M * N * (double)K * batch, s);
}

cudaError_t dgemm_views(int M, int N, int K, double alpha, const KView& A, const KView& B,
                        double beta, double* C, long ldc, cudaStream_t s, bool sym) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (sym && (M != N || beta != 0.0)) return cudaErrorInvalidValue;
  const long straight = (long)((M + 7) / 8) * ((N + 31) / 32);
  const long turned = (long)((N + 7) / 8) * ((M + 31) / 32);
  const bool t = turned < straight;
  const KView &a = t ? B : A, &b = t ? A : B;
  GemmArgs g{};
  g.M = t ? N : M;
  g.N = t ? M : N;
  g.K = K;
  g.alpha = alpha;
  g.beta = beta;
  g.A = a.X; g.ai = a.rs; g.ak = a.cs; g.akin = (unsigned)a.kin; g.akout = a.kout;
  g.B = b.X; g.bj = b.rs; g.bk = b.cs; g.bkin = (unsigned)b.kin; g.bkout = b.kout;
  g.C = C; g.ci = t ? 1 : ldc; g.cj = t ? ldc : 1;
  g.tn = (g.N + kGT - 1) / kGT;
  g.sym = sym ? 1 : 0;
  const long tiles = sym ? (long)g.tn * (g.tn + 1) / 2 : (long)((g.M + kGT - 1) / kGT) * g.tn;
  return launch_dgemm(g, tiles, 1, 2.0 * M * N * (double)K, s);
}

cudaError_t dgemm_sym(int N, int K, double alpha, const double* A, int lda, bool ta,
                      const double* B, int ldb, bool tb, double beta, double* C, int ldc,
                      cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  GemmArgs g{};
  g.M = N; g.N = N; g.K = K;
  g.alpha = alpha;
  g.beta = beta;
  g.A = A; g.ai = ta ? 1 : lda; g.ak = ta ? lda : 1;
  g.B = B; g.bk = tb ? 1 : ldb; g.bj = tb ? ldb : 1;
  g.C = C; g.ci = ldc; g.cj = 1;
  g.sym = 1;
  g.tn = (N + kGT - 1) / kGT;
  const long tiles = (long)g.tn * (g.tn + 1) / 2;
  return launch_dgemm(g, tiles, 1, 2.0 * kGT * kGT * (double)K * (double)tiles, s);
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
