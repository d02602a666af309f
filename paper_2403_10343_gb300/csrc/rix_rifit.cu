// RI-LVL coefficient fit (the paper's Eq. 8 with the pair-restricted Coulomb
// metric of Eq. 10; the "Initialization" stage of the exchange build):
//
//   C^mu_ij = sum_{nu in P(IJ)} (ij|nu) L^{IJ}_{nu mu},   L^{IJ} = (V^{IJ})^{-1},
//
// for every atom pair (I, J, n), with P(IJ) = aux(I) u aux(J) (aux(I) alone for
// the on-site pair) and V^{IJ} the Coulomb matrix restricted to P(IJ): the
// on-site blocks V(I,I,0), V(J,J,0) on the diagonal and V(I,J,n) off it.  Each
// representative pair (I < J, or I == J with n > 0, or on-site) is factored by
// one CTA: V^{IJ} + lambda 1 = L D L^T (L unit lower triangular; right-looking, a
// barrier per column).  Then warps solve L D L^T x = (ij|.), one (i, j) column per
// lane, and the partner pair (J, I, -n) receives the same numbers with (i, j)
// and the two aux sets swapped, so the fitted C is exactly pair symmetric.
// lambda > 0 shifts the diagonal (a Tikhonov fit) for metrics that are
// numerically singular.
//
// The n^2 nb_I nb_J multiply-adds of the two triangular solves are most of the work (the
// FP64 pipe is the bound).  They are spread as units of 32 columns of equal length (of one pair or
// the next ones of the same size), longest first, so that every lane has work and pairs of any
// size fill the chip together (a pair of O has 196 columns of 112 functions, a pair of H 25 of 32); a lane takes eight rows at a time, so that a value of x read back serves eight
// multiply-adds, and L streams through L1 (3.5 KB per eight rows, the same for all lanes).
// ((H2O)27, 3,321 pairs: 6.04 ms with a CTA of 256 per pair for everything, a row at a time; 4.62 ms
// with eight rows and the triangle in shared memory; 2.84 ms now.)
#include <algorithm>
#include <vector>

#include "rix_internal.h"

namespace {

constexpr int FIT_RB = 8;                  // rows of a solve at a time
constexpr int FIT_SMEM = 100 * 1024;       // largest triangle factored in shared memory
constexpr int FIT_MAXN = 512;              // two aux sets of 256

__device__ __forceinline__ int64_t tri(int i) { return (int64_t)i * (i + 1) / 2; }  // start of row i

// lower triangle of M = V^{IJ} + lambda 1 for pair p (n x n, packed by rows)
__device__ void assemble(double *M, int n, int naA, int naB, const double *Vaa, const double *Vbb, const double *Vab,
                         double lambda) {
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int r = e / n, c = e - r * n;
    if (c > r) continue;
    const double v = r < naA ? Vaa[r * naA + c] : c >= naA ? Vbb[(r - naA) * naB + (c - naA)] : Vab[c * naB + (r - naA)];
    M[tri(r) + c] = r == c ? v + lambda : v;
  }
}

// rows [i0, i0 + nr) of column col: y = L^-1 b (rows before i0 of y in x)
template <int NR>
__device__ __forceinline__ void forward_rows(const double *M, const double *rhs, double *x, int cols, int col, int i0,
                                             int nr) {
  double acc[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = r < nr ? rhs[(int64_t)(i0 + r) * cols + col] : 0.0;
  const double *row[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) row[r] = M + tri(i0 + (r < nr ? r : 0));
#pragma unroll 4
  for (int j = 0; j < i0; j++) {
    const double xj = x[(int64_t)j * cols + col];
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r] = fma(-row[r][j], xj, acc[r]);
  }
#pragma unroll
  for (int r = 0; r < NR; r++) {
    if (r < nr) {
#pragma unroll
      for (int q = 0; q < r; q++) acc[r] = fma(-row[r][i0 + q], acc[q], acc[r]);
      x[(int64_t)(i0 + r) * cols + col] = acc[r];
    }
  }
}

// rows [i0, i0 + nr): x = L^-T D^-1 y (rows from i0 + nr on already solved)
template <int NR>
__device__ __forceinline__ void backward_rows(const double *M, const double *rd, double *x, int n, int cols, int col,
                                              int i0, int nr) {
  double acc[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = r < nr ? x[(int64_t)(i0 + r) * cols + col] * rd[i0 + r] : 0.0;
#pragma unroll 2
  for (int j = i0 + nr; j < n; j++) {
    const double xj = x[(int64_t)j * cols + col];
    const double *lj = M + tri(j) + i0;
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r] = fma(-lj[r], xj, acc[r]);  // (r >= nr: row j's next entries, not used)
  }
#pragma unroll
  for (int r = NR - 1; r >= 0; r--) {
    if (r < nr) {
#pragma unroll
      for (int q = r + 1; q < NR; q++)
        if (q < nr) acc[r] = fma(-M[tri(i0 + q) + i0 + r], acc[q], acc[r]);
      x[(int64_t)(i0 + r) * cols + col] = acc[r];
    }
  }
}

// L (packed by rows, the unit diagonal not stored as such) and 1/D behind it, per pair in work
template <bool SHARED>
__global__ void __launch_bounds__(256)
    k_rifit_factor(const int32_t *rep, const int32_t *pA, const int32_t *pB, const uint8_t *onsite,
                   const int32_t *onsite_pair, const int32_t *na, const double *__restrict__ V, const int64_t *offV,
                   double lambda, double *work, const int64_t *woff, int *err) {
  extern __shared__ double tri_sm[];
  const int p = rep[blockIdx.x];
  const int a = pA[p], b = pB[p];
  const int naA = na[a], naB = na[b];
  const int n = naA + (onsite[p] ? 0 : naB);
  double *L = work + woff[blockIdx.x], *rd = L + tri(n);
  double *M = SHARED ? tri_sm : L;
  assemble(M, n, naA, naB, V + offV[onsite_pair[a]], V + offV[onsite_pair[b]], V + offV[p], lambda);
  __syncthreads();
  // After step k column k holds L D (its diagonal D) and the trailing triangle is updated; the
  // thread that updates the next pivot takes its reciprocal, so a step needs one barrier and the
  // other warps do not repeat the division (ten FP64 instructions of 64 clocks each).  Eight
  // lanes to a row: most rows of the triangle are short.
  __shared__ double srd[FIT_MAXN];
  const int g8 = threadIdx.x >> 3, l8 = threadIdx.x & 7, n8 = blockDim.x >> 3;
  bool bad = false;  // thread 0 takes every pivot
  auto pivot = [&](int k) {
    const double d = M[tri(k) + k];
    if (!(d > 0.0)) bad = true;
    srd[k] = 1.0 / (d > 0.0 ? d : 1.0);
  };
  if (threadIdx.x == 0) pivot(0);
  __syncthreads();
  for (int k = 0; k < n - 1; k++) {
    const double r = srd[k];
    for (int i = k + 1 + g8; i < n; i += n8) {
      double *mi = M + tri(i);
      const double f = -mi[k] * r;
      for (int j = k + 1 + l8; j <= i; j += 8) mi[j] = fma(f, M[tri(j) + k], mi[j]);
    }
    if (threadIdx.x == 0) pivot(k + 1);  // row k + 1 is thread 0's alone
    __syncthreads();
  }
  if (bad) atomicExch(err, 1);
  for (int i = g8; i < n; i += n8) {
    if (l8 == 0) rd[i] = srd[i];
    for (int k = l8; k < i; k += 8) L[tri(i) + k] = M[tri(i) + k] * srd[k];
  }
}

// One column per lane: a unit is 32 columns from column y of pair x on, running on into the next
// pairs as long as their metric has the same size.  Forward then backward substitution in place in C(p),
// then the partner (B, A, -n): C(q)[mu'][j][i] = C(p)[mu][i][j], mu' = mu with the aux sets swapped.
__global__ void __launch_bounds__(64)
    k_rifit_solve(int64_t nunits, const int2 *units, int rend, const int32_t *rep, const int32_t *pA, const int32_t *pB,
                  const int32_t *partner, const uint8_t *onsite, const int32_t *nb, const int32_t *na,
                  const double *__restrict__ eri, const int64_t *offC, const double *__restrict__ work,
                  const int64_t *woff, double *C) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= nunits) return;
  const int2 u = units[w];
  auto size = [&](int r) {
    const int p = rep[r];
    return na[pA[p]] + (onsite[p] ? 0 : na[pB[p]]);
  };
  const int n = size(u.x);
  int r = u.x, col = u.y + (threadIdx.x & 31);
  while (r < rend && size(r) == n) {
    const int c = nb[pA[rep[r]]] * nb[pB[rep[r]]];
    if (col < c) break;
    col -= c;
    r++;
  }
  if (r >= rend || size(r) != n) return;
  const int p = rep[r];
  const int a = pA[p], b = pB[p];
  const bool ons = onsite[p];
  const int naA = na[a], naB = na[b], nbA = nb[a], nbB = nb[b], cols = nbA * nbB;
  const double *M = work + woff[r], *rd = M + tri(n);
  const double *rhs = eri + offC[p];
  double *x = C + offC[p];
  const int full = n / FIT_RB * FIT_RB;
  for (int i0 = 0; i0 < full; i0 += FIT_RB) forward_rows<FIT_RB>(M, rhs, x, cols, col, i0, FIT_RB);
  for (int i0 = full; i0 < n; i0++) forward_rows<1>(M, rhs, x, cols, col, i0, 1);
  for (int i0 = n - 1; i0 >= full; i0--) backward_rows<1>(M, rd, x, n, cols, col, i0, 1);
  for (int i0 = full - FIT_RB; i0 >= 0; i0 -= FIT_RB) backward_rows<FIT_RB>(M, rd, x, n, cols, col, i0, FIT_RB);
  if (ons) return;
  double *y = C + offC[partner[p]];
  const int i = col / nbB, j = col - i * nbB;
  for (int mu = 0; mu < n; mu++) {
    const int mq = mu < naA ? naB + mu : mu - naA;
    y[((int64_t)mq * nbB + j) * nbA + i] = x[(int64_t)mu * cols + col];
  }
}

}  // namespace

extern "C" rix_status rix_fit_C(rix_ctx *ctx, const double *V, const double *eri, double lambda, double *C,
                                void *stream) {
  if (!ctx || !V || !eri || !C || !(lambda >= 0.0)) return RIX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  // representative pairs, their metric sizes, and the on-site pair of every atom
  std::vector<int32_t> rep, ons(ctx->nat, -1);
  for (int64_t p = 0; p < ctx->np; p++) {
    const int a = ctx->pA[p], b = ctx->pB[p];
    if (ctx->onsite[p]) ons[a] = (int32_t)p;
    bool is_rep = ctx->onsite[p] || a < b;
    if (a == b && !ctx->onsite[p]) {
      const int8_t *n = &ctx->pn[3 * p];
      is_rep = n[0] > 0 || (n[0] == 0 && (n[1] > 0 || (n[1] == 0 && n[2] > 0)));
    }
    if (is_rep) rep.push_back((int32_t)p);
  }
  for (int a = 0; a < ctx->nat; a++)
    if (ons[a] < 0) {
      ctx->last_error = "rix_fit_C: an atom without its on-site pair";
      return RIX_EINVAL;
    }
  // pairs in the order of their work, so the long ones start first; metrics above the shared-memory
  // limit (in the workspace throughout) come before the others
  auto metric_n = [&](int p) { return (int64_t)ctx->na_at[ctx->pA[p]] + (ctx->onsite[p] ? 0 : ctx->na_at[ctx->pB[p]]); };
  auto big = [&](int p) { return metric_n(p) * (metric_n(p) + 1) / 2 * 8 > FIT_SMEM; };
  std::stable_sort(rep.begin(), rep.end(), [&](int32_t x, int32_t y) { return metric_n(x) > metric_n(y); });
  // batches whose factors fit a 1 GB workspace; per batch the solve units, 32 columns each
  const int64_t budget = (int64_t)1 << 27;  // doubles
  struct Batch {
    size_t first, mid, last;  // [first, mid): factored in the workspace
    size_t u0, u1;
    int smem;
  };
  std::vector<Batch> batches;
  std::vector<int64_t> woff(rep.size(), 0);
  std::vector<int2> units;
  int64_t maxw = 0;
  for (size_t r = 0; r < rep.size();) {
    Batch bt{r, r, r, units.size(), 0, 0};
    int64_t w = 0;
    int next = 0;  // first column of the next unit in the pair at hand
    for (; bt.last < rep.size(); bt.last++) {
      const int p = rep[bt.last];
      const int64_t n = metric_n(p), sz = n * (n + 1) / 2 + n;
      if (w > 0 && w + sz > budget) break;
      woff[bt.last] = w;
      w += sz;
      if (big(p)) bt.mid = bt.last + 1;
      else bt.smem = std::max(bt.smem, (int)(n * (n + 1) / 2 * 8));
      if (bt.last == r || n != metric_n(rep[bt.last - 1])) next = 0;  // a new size starts a new unit
      const int cols = ctx->nb_at[ctx->pA[p]] * ctx->nb_at[ctx->pB[p]];
      for (; next < cols; next += 32) units.push_back(make_int2((int)bt.last, next));
      next -= cols;
    }
    bt.u1 = units.size();
    maxw = std::max(maxw, w);
    batches.push_back(bt);
    r = bt.last;
  }
  int32_t *d_rep = nullptr, *d_ons = nullptr;
  int64_t *d_woff = nullptr;
  int2 *d_units = nullptr;
  double *d_work = nullptr;
  int *d_err = nullptr;
  cudaError_t e = cudaFuncSetAttribute(k_rifit_factor<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FIT_SMEM);
  auto alloc = [&](void **p, size_t bytes) {
    if (e == cudaSuccess) e = cudaMallocAsync(p, bytes, st);
  };
  auto put = [&](void *d, const void *h, size_t bytes) {
    if (e == cudaSuccess) e = cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, st);
  };
  alloc((void **)&d_rep, sizeof(int32_t) * std::max<size_t>(rep.size(), 1));
  alloc((void **)&d_ons, sizeof(int32_t) * ctx->nat);
  alloc((void **)&d_woff, sizeof(int64_t) * std::max<size_t>(rep.size(), 1));
  alloc((void **)&d_units, sizeof(int2) * std::max<size_t>(units.size(), 1));
  alloc((void **)&d_work, sizeof(double) * std::max<int64_t>(maxw, 1));
  alloc((void **)&d_err, sizeof(int));
  put(d_rep, rep.data(), sizeof(int32_t) * rep.size());
  put(d_ons, ons.data(), sizeof(int32_t) * ctx->nat);
  put(d_woff, woff.data(), sizeof(int64_t) * rep.size());
  put(d_units, units.data(), sizeof(int2) * units.size());
  if (e == cudaSuccess) e = cudaMemsetAsync(d_err, 0, sizeof(int), st);
  for (const Batch &bt : batches) {
    if (e != cudaSuccess) break;
    auto factor = [&](auto *kernel, size_t r0, size_t r1, int smem) {
      if (r1 > r0 && e == cudaSuccess) {
        kernel<<<(unsigned)(r1 - r0), 256, smem, st>>>(d_rep + r0, ctx->d_pA, ctx->d_pB, ctx->d_onsite, d_ons, ctx->d_na,
                                                       V, ctx->d_offV, lambda, d_work, d_woff + r0, d_err);
        e = cudaGetLastError();
      }
    };
    factor(k_rifit_factor<false>, bt.first, bt.mid, 0);
    factor(k_rifit_factor<true>, bt.mid, bt.last, bt.smem);
    if (e != cudaSuccess) break;
    const int64_t nu = (int64_t)(bt.u1 - bt.u0);
    k_rifit_solve<<<(unsigned)((nu + 1) / 2), 64, 0, st>>>(nu, d_units + bt.u0, (int)bt.last, d_rep, ctx->d_pA, ctx->d_pB,
                                                           ctx->d_partner1, ctx->d_onsite, ctx->d_nb, ctx->d_na, eri,
                                                           ctx->d_offC, d_work, d_woff, C);
    e = cudaGetLastError();
  }
  int herr = 0;
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = cudaMemcpy(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost);
  for (void *p : {(void *)d_rep, (void *)d_ons, (void *)d_woff, (void *)d_units, (void *)d_work, (void *)d_err})
    if (p) cudaFreeAsync(p, st);
  if (e != cudaSuccess) {
    ctx->last_error = std::string("rix_fit_C: ") + cudaGetErrorString(e);
    return RIX_ECUDA;
  }
  if (herr) {
    ctx->last_error = "rix_fit_C: a pair's Coulomb metric is not positive definite (raise lambda)";
    return RIX_EINVAL;
  }
  return RIX_OK;
}
