// FP64 path of the exchange build and the shared small kernels.
//
// The build runs the paper's grouping of the RI-LVL sum by the atoms that
// carry the two auxiliary functions (Eq. 11, Eqs. 12a-12d).  With i on A, j on B',
// k on G', l on E' it computes
//
//   T(A,G')   = sum_B' C(A,B')^{P on A} D(B',G')                (E = C*D)
//   U2(A,G')  = V(A,G')^T T(A,G')                               (G = E'*V)
//   X(A,E')   = 1/2 sum_G' [V(A,E')^T T(A,G')]^{Q on E'} C(G',E')^{Q on E'}   term 1
//             +     sum_G'!=E' U2(A,G') C(G',E')^{Q on G'}                     term 2
//   Z(B,E')   = 1/2 sum_G'!=E' [V(B,G') C(G',E')^{Q on G'}] applied to D(B,G') (H = F*D)
//               (or over the unordered pairs {B,G'}: rix_ctx::wZ)
//   X(A,E')  +=     sum_B'!=A C(A,B')^{P on B'} Z(B,E')                        term 4
//   K(A,E',n) = X(A,E',n) + X(E',A,-n)^T
//
// Term 3 (P on B', Q on E') equals term 2 transposed (the pair symmetry of C,
// V and D stated after Eqs. 12a-12d; the paper's "2G"), and terms 1 and 4 are symmetric by
// themselves, so the last line restores all four terms exactly.
//
// Each kernel is output-stationary: one CTA (or a cluster of them) owns an output
// block or a row tile of it, walks its product list and keeps the sums in registers, so no
// atomics are needed and every run sums in the same order.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>
#include <string>

#include "rix_internal.h"

using namespace rix;
namespace cg = cooperative_groups;

namespace {

constexpr int NT = 256;      // threads per CTA
constexpr int MAXE = 32;     // output elements per thread in tiled kernels
static_assert(NT * MAXE == CAP_MAX, "row tiles");
constexpr int XMAXE = 16;    // output elements per thread for K blocks above 256 elements (64 x 64 / 256)
constexpr int SM_MAX = 16384;  // largest shared-memory tile budget in doubles (128 KB)

// ------------------------------------------------------------------ pair list (a1)
__device__ __forceinline__ double d2_raw(const double *xyz, const double *cell, int periodic, int a, int b,
                                         int n1, int n2, int n3) {
  double s[3] = {0.0, 0.0, 0.0};
  if (periodic) {
#pragma unroll
    for (int c = 0; c < 3; c++)
      s[c] = __dadd_rn(__dadd_rn(__dmul_rn((double)n1, cell[c]), __dmul_rn((double)n2, cell[3 + c])),
                       __dmul_rn((double)n3, cell[6 + c]));
  }
  double dx[3];
#pragma unroll
  for (int c = 0; c < 3; c++) dx[c] = __dsub_rn(__dadd_rn(xyz[3 * b + c], s[c]), xyz[3 * a + c]);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx[0], dx[0]), __dmul_rn(dx[1], dx[1])), __dmul_rn(dx[2], dx[2]));
}

__device__ __forceinline__ bool is_rep(int a, int b, int n1, int n2, int n3) {
  if (a != b) return a < b;
  if (n1 != 0) return n1 > 0;
  if (n2 != 0) return n2 > 0;
  return n3 >= 0;
}

// One warp per atom A; candidates (B, n1, n2, n3) in lexicographic order, so
// the kept pairs come out sorted.  Pass 1 counts, pass 2 writes the keys.
__global__ void k_pairs(int nat, const double *xyz, const double *cell, int periodic, int nr0, int nr1,
                        int nr2, double rc2, int cut, int64_t *counts, const int64_t *rowptr, int64_t *keys) {
  int warp = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  int lane = threadIdx.x & 31;
  if (warp >= nat) return;
  const int a = warp;
  const int N1 = 2 * nr0 + 1, N2 = 2 * nr1 + 1, N3 = 2 * nr2 + 1;
  const int64_t total = (int64_t)nat * N1 * N2 * N3;
  int64_t pos = rowptr ? rowptr[a] : 0;
  int64_t cnt = 0;
  for (int64_t base = 0; base < total; base += 32) {
    int64_t c = base + lane;
    bool keep = false;
    int b = 0, n1 = 0, n2 = 0, n3 = 0;
    if (c < total) {
      int64_t r = c;
      n3 = (int)(r % N3) - nr2; r /= N3;
      n2 = (int)(r % N2) - nr1; r /= N2;
      n1 = (int)(r % N1) - nr0; r /= N1;
      b = (int)r;
      if (!cut) {
        keep = true;
      } else {
        double d2 = is_rep(a, b, n1, n2, n3) ? d2_raw(xyz, cell, periodic, a, b, n1, n2, n3)
                                             : d2_raw(xyz, cell, periodic, b, a, -n1, -n2, -n3);
        keep = d2 < rc2;
      }
    }
    unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keys && keep) keys[pos + __popc(m & ((1u << lane) - 1u))] = pair_key(a, b, n1, n2, n3);
    pos += __popc(m);
    cnt += __popc(m);
  }
  if (counts && lane == 0) counts[a] = cnt;
}

// ------------------------------------------------------------------ screening flags
// keep[b] = max |block b| >= tau (always 1 when tau <= 0); one CTA of W warps per block.
// norm (optional): the block's max |x| rounded up to a float (product screening).  C and V blocks
// (up to 176 KB) take eight warps, D blocks (at most 1.5 KB in the water systems) one.
template <int W>
__global__ void __launch_bounds__(256)
    k_flags(const double *arr, const int64_t *off, int64_t n, double tau, uint8_t *keep, float *norm) {
  // W == 1: eight blocks to a CTA
  const int64_t w = W == 1 ? (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5 : blockIdx.x;
  const int t = W == 1 ? threadIdx.x & 31 : threadIdx.x;
  if (w >= n) return;
  if (!(tau > 0) && !norm) {
    if (t == 0) keep[w] = 1;
    return;
  }
  double m = 0;
#pragma unroll 4
  for (int64_t i = off[w] + t; i < off[w + 1]; i += 32 * W) m = fmax(m, fabs(arr[i]));
  for (int s = 16; s; s >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, s));
  if (W > 1) {
    __shared__ double red[W];
    if ((t & 31) == 0) red[t >> 5] = m;
    __syncthreads();
    if (t == 0)
      for (int i = 1; i < W; i++) m = fmax(m, red[i]);
  }
  if (t == 0) {
    keep[w] = !(tau > 0) || m >= tau;
    if (norm) norm[w] = __double2float_ru(m);
  }
}

// ------------------------------------------------------------------ symmetry check of C and V
// C(B,A,-n)[P'][j][i] == C(A,B,n)[P][i][j] with P' the same aux function, and
// V(B,A,-n) == V(A,B,n)^T, bit for bit.  One CTA per pair, which compares both of the two partners
// (each comparison is its own mirror); sets *flag on a mismatch.  ((H2O)27: 325 us with a warp
// per pair, both partners comparing; 78 us now.)
__global__ void __launch_bounds__(256)
    k_symcheck(const int32_t *pA, const int32_t *pB, const int32_t *partner, const uint8_t *onsite, const int32_t *nb,
               const int32_t *na, const double *C, const int64_t *offC, const double *V, const int64_t *offV,
               int32_t *flag) {
  const int64_t p = blockIdx.x;
  const int64_t q = partner[p];
  if (q < p) return;
  const int a = pA[p], b = pB[p];
  const int nbA = nb[a], nbB = nb[b], naA = na[a], naB = na[b];
  const bool ons = onsite[p];
  bool bad = false;
  const double *c = C + offC[p], *cq = C + offC[q];
  const int n = (naA + (ons ? 0 : naB)) * nbA * nbB;
#pragma unroll 4
  for (int e = threadIdx.x; e < n; e += 256) {
    const int P = e / (nbA * nbB), r = e - P * (nbA * nbB);
    const int i = r / nbB, j = r - i * nbB;
    const int Pq = ons ? P : (P < naA ? P + naB : P - naA);
    bad |= c[e] != cq[(Pq * nbB + j) * nbA + i];
  }
  const double *v = V + offV[p], *vq = V + offV[q];
  for (int e = threadIdx.x; e < naA * naB; e += 256) {
    const int P = e / naB, Q = e - P * naB;
    bad |= v[e] != vq[Q * naA + P];
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

// ------------------------------------------------------------------ live blocks
// live[t] = 1 when a product of the list of block t is kept: T(A,G') <- (C(A,B'), D(B',G')) with
// L the T list, Z(B,E') <- (pair (B,G'), pair (G',E')) with the Z list (keepV given).  The other
// blocks are zero, and the kernels that read T or Z skip them (in the 24-atom ice cell, whose D
// reaches a quarter of the pairs, half of the terms-3+4 products).  One warp per block.
__global__ void k_live(int64_t n, const int64_t *ptr, const int2 *L, const uint8_t *keepC, const uint8_t *keepV,
                       const uint8_t *keepD, PScreen ps, uint8_t *live) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= n) return;
  bool any = false;
  for (int64_t e = ptr[t]; e < ptr[t + 1] && !any; e += 32) {
    bool k = false;
    if (e + lane < ptr[t + 1]) {
      const int2 en = L[e + lane];
      k = keepV ? keepD[en.x] && keepV[en.x] && keepC[en.y] && !ps.drop3(en.x, en.x, en.y)
                : keepC[en.x] && keepD[en.y] && !ps.drop2(en.x, en.y);
    }
    any = __any_sync(0xffffffffu, k);
  }
  if (lane == 0) live[t] = any;
}

// ------------------------------------------------------------------ stage T
// T(A,G')[P][i][k] for P in [p0, p0+pt): sum over (C(A,B'), D(B',G')) entries.  The contraction
// columns (B', j) of the kept entries are taken TCOL at a time: one warp makes a table of their C
// offsets, all threads stage the D rows, and every element sums over the whole batch between two
// barriers (an entry alone is 5 or 14 multiply-adds per element, less than its barriers cost).
// (H2O)64: 110 -> 82 ms (1.16 TFLOP/s of 1.25).
constexpr int TCOL = 128;   // columns of a batch at most (an entry has up to 64)
struct TCols {
  int64_t c[TCOL], d[TCOL];  // offsets of C(A,B')[0][0][j] and D(B',G')[j][0]
  int nb[TCOL];              // nb of B' (row stride of C)
  int n, next;               // columns; entries taken
};

__global__ void __launch_bounds__(NT) k_T(const int2 *items, const int64_t *ptrT, const int2 *LT,
                                          const int32_t *atomA2, const int32_t *atomB2, const int64_t *off2,
                                          const int32_t *pB, const int32_t *nb, const int32_t *na,
                                          const double *__restrict__ C, const int64_t *offC,
                                          const double *__restrict__ D, const int64_t *offD,
                                          const uint8_t *keepC, const uint8_t *keepD, double *T,
                                          int64_t tbase, const uint8_t *ttc, int cap, PScreen ps) {
  extern __shared__ double sm[];
  __shared__ TCols tb;
  const int tid = threadIdx.x;
  const int2 it = items[blockIdx.x];
  const int t = it.x, p0 = it.y;
  const int a = atomA2[t], g = atomB2[t];
  if (ttc && ttc[a]) return;  // this row atom's T comes from the tensor cores
  const int nbA = nb[a], naA = na[a], nbG = nb[g];
  const int per = nbA * nbG;
  const int pt = max(1, cap / per);
  const int pe = min(naA, p0 + pt);
  const int nel = (pe - p0) * per;
  double acc[MAXE];
#pragma unroll
  for (int r = 0; r < MAXE; r++) acc[r] = 0.0;
  for (int64_t e = ptrT[t]; e < ptrT[t + 1];) {
    __syncthreads();
    if (tid < 32) {
      const bool in = e + tid < ptrT[t + 1];
      const int2 en = LT[in ? e + tid : e];
      const int w = in && keepC[en.x] && keepD[en.y] && !ps.drop2(en.x, en.y) ? nb[pB[en.x]] : 0;
      int s = w;  // columns up to and including this entry's
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, s, o);
        if (tid >= o) s += v;
      }
      const int take = __popc(__ballot_sync(0xffffffffu, in && s <= TCOL));
      if (tid < take) {
        const int64_t c0 = offC[en.x] + (int64_t)p0 * nbA * w, d0 = offD[en.y];
        for (int j = 0; j < w; j++) {
          tb.c[s - w + j] = c0 + j;
          tb.d[s - w + j] = d0 + j * nbG;
          tb.nb[s - w + j] = w;
        }
      }
      if (tid == take - 1) {
        tb.n = s;
        tb.next = take;
      }
    }
    __syncthreads();
    const int n = tb.n;
    e += tb.next;
    if (n == 0) continue;
    for (int i = tid; i < n * nbG; i += NT) {
      const int c = i / nbG;
      sm[i] = __ldg(D + tb.d[c] + (i - c * nbG));
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < MAXE; r++) {
      const int el = tid + r * NT;
      if (el < nel) {
        const int row = el / nbG;
        const double *dc = sm + (el - row * nbG);
        double s = acc[r];
#pragma unroll 4
        for (int c = 0; c < n; c++) s = fma(__ldg(C + tb.c[c] + row * tb.nb[c]), dc[c * nbG], s);
        acc[r] = s;
      }
    }
  }
  double *out = T + (off2[t] - tbase) + (int64_t)p0 * per;
#pragma unroll
  for (int r = 0; r < MAXE; r++) {
    const int el = tid + r * NT;
    if (el < nel) out[el] = acc[r];
  }
}

// ------------------------------------------------------------------ stage U2
// U2(A,G')[Q][i][k] = sum_P V(A,G')[P][Q] T(A,G')[P][i][k] for Q in [q0, q0+qt).
__global__ void __launch_bounds__(NT) k_U2(const int2 *items, const int32_t *pA, const int32_t *pB,
                                           const int32_t *nb, const int32_t *na, const double *__restrict__ V,
                                           const int64_t *offV, const uint8_t *keepV, const int32_t *map1to2,
                                           const double *__restrict__ T, const int64_t *off2,
                                           const int64_t *offU, double *U, int64_t tbase, int cap) {
  const int2 it = items[blockIdx.x];
  const int p = it.x, q0 = it.y;
  if (!keepV[p]) return;
  const int a = pA[p], g = pB[p];
  const int nbA = nb[a], naA = na[a], nbG = nb[g], naG = na[g];
  const int per = nbA * nbG;
  const int qt = max(1, cap / per);
  const int qe = min(naG, q0 + qt);
  const int nel = (qe - q0) * per;
  const double *Vb = V + offV[p];
  const double *Tt = T + (off2[map1to2[p]] - tbase);
  double *out = U + offU[p] + (int64_t)q0 * per;
  for (int el = threadIdx.x; el < nel; el += NT) {
    const int q = q0 + el / per, c = el % per;
    double s = 0.0;
    for (int P = 0; P < naA; P++) s = fma(__ldg(Vb + P * naG + q), __ldg(Tt + (int64_t)P * per + c), s);
    out[el] = s;
  }
}

// ------------------------------------------------------------------ K-block outputs (terms 1+2, terms 3+4)
// A K block has few elements (196 for a pair of O, 25 for a pair of H) and sums
// long products, so a CTA splits the contraction and not only the output:
// thread tid works on element tid % nel in group tid / nel, each group sums its own
// share of every product, and the shares are added in a fixed order at the end.  Two
// DFMA per clock and SM leave 64 clocks to a warp instruction, so what counts is
// that every lane has work and that warps of several CTAs overlap the loads; the
// products that need no staging run without a barrier.  Where a system has few or very
// uneven outputs, a cluster of ns CTAs shares one output (the launch classes of rix_ctx).
// R elements per thread: 1 up to 256 elements, else 16 (and one group).
// GB300, one group with staged operands, with these kernels at first, and now with the cheaper
// orientation of term 1 and empty T and Z blocks skipped: (H2O)64 terms 1+2 652, 309 and 267 ms (1.15
// TFLOP/s of the products it keeps, FP64 pipe 1.25), 24-atom ice cell terms 3+4 245, 115 and
// 61 ms; (H2O)8, split over 2^c CTAs, terms 1+2 5.34, 1.99 and 1.75 ms.  K blocks above 256 elements (12-atom
// perovskite, up to 1,521): the whole FP64 build 1,483 and 700 ms.
struct Split {
  int ng, grp, el0;  // groups of the CTA, this thread's group (ng: no work) and first element
  int part, parts;   // share of this thread's group among the shares of the whole cluster
};

template <int R>
__device__ __forceinline__ Split split_of(int nel, int rank, int ns) {
  Split s;
  s.ng = R == 1 ? NT / nel : 1;
  s.grp = R == 1 ? (int)threadIdx.x / nel : 0;
  s.el0 = R == 1 ? (int)threadIdx.x - s.grp * nel : (int)threadIdx.x;
  s.part = rank * s.ng + s.grp;
  s.parts = ns * s.ng;
  return s;
}

// acc[r] += sum over this share of the rows (P, j) of a[P][i][j] b[P][j][l] (a: nP x nbA x nbJ,
// b: nP x nbJ x nbE); element el = i nbE + l.  The share is summed by itself before it is added:
// sums of sums round less than one long chain ((H2O)64, terms 1-4 together: relative error of K
// 9.5e-15 -> 1.1e-15 for 657 -> 660 ms).
template <int R>
__device__ __forceinline__ void dot_share(double (&acc)[R], const Split &s, int nel, const double *__restrict__ a,
                                          const double *__restrict__ b, int nP, int nbA, int nbJ, int nbE) {
  if (s.grp >= s.ng) return;
  const int K = nP * nbJ;
  const int k0 = (int)((int64_t)K * s.part / s.parts), k1 = (int)((int64_t)K * (s.part + 1) / s.parts);
  const int P0 = k0 / nbJ, j0 = k0 - P0 * nbJ;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int el = s.el0 + r * NT;
    if (el < nel) {
      const int i = el / nbE, l = el - i * nbE;
      const double *ap = a + ((int64_t)P0 * nbA + i) * nbJ + j0;
      const double *bp = b + (int64_t)k0 * nbE + l;
      double v = 0.0;
      int j = j0;
#pragma unroll 4
      for (int k = k0; k < k1; k++) {
        v = fma(__ldg(ap), __ldg(bp), v);
        bp += nbE;
        ap++;
        if (++j == nbJ) {  // the next P: same row i
          j = 0;
          ap += (nbA - 1) * nbJ;
        }
      }
      acc[r] += v;
    }
  }
}

// The sum of all shares of a cluster's output, in rank 0: groups first, then ranks.
// red: NT (R == 1) or nel doubles of shared memory.
template <int R, class F>
__device__ __forceinline__ void gather_shares(double (&acc)[R], const Split &s, int nel, int ns, double *red, F store) {
  if (R == 1 && s.ng > 1) {
    __syncthreads();
    red[threadIdx.x] = acc[0];
    __syncthreads();
    if ((int)threadIdx.x < nel) {
      double v = acc[0];
      for (int g = 1; g < s.ng; g++) v += red[g * nel + threadIdx.x];
      acc[0] = v;
    }
  }
  if (ns > 1) {
    cg::cluster_group cl = cg::this_cluster();
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int el = threadIdx.x + r * NT;
      if (el < nel) red[el] = acc[r];
    }
    cl.sync();
    if (cl.block_rank() == 0) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int el = threadIdx.x + r * NT;
        if (el < nel)
          for (int q = 1; q < ns; q++) acc[r] += cl.map_shared_rank(red, q)[el];
      }
    }
    cl.sync();
    if (cl.block_rank() != 0) return;
  }
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int el = threadIdx.x + r * NT;
    if (el < nel) store(el, acc[r]);
  }
}

// ------------------------------------------------------------------ terms 1 and 2
// Term 1, U1[Q][i][k] = sum_P V(A,E')[P][Q] T(A,G')[P][i][k] (Q on E') and X += U1 C(G',E'), takes
// the columns (G', k) of several entries at once: a table of the columns' T and C offsets, U1 of a
// few Q over all of them in shared memory (full warps whatever the species), then the split product.
// Term 2 is a split product per entry.
constexpr int XCOL = 192;    // columns of a batch at most
struct XCols {
  int64_t t[XCOL], c[XCOL];  // offsets of T(A,G')[0][0][k] and C(G',E')[Q = 0 on E'][k][0]
  int nb[XCOL];              // nb of G'
  int n, next;               // columns; first list entry after the batch
};

// XCols of the list entries from it on that term 1 uses, at most maxcol columns (one warp)
__device__ __forceinline__ void x12_batch(XCols &tb, int64_t it, int64_t end, int maxcol, const X12Entry *L,
                                          const uint8_t *keepC, const int32_t *pA, const int32_t *nb,
                                          const int32_t *na, const uint8_t *onsite, const int64_t *off2,
                                          int64_t tbase, const int64_t *offC, int nbE, const uint8_t *liveT) {
  const int lane = threadIdx.x & 31;
  const bool in = it + lane < end;
  const X12Entry en = L[in ? it + lane : it];
  const int g = pA[en.p3];
  const int w = in && en.t1 && keepC[en.p3] && !(liveT && !liveT[en.t]) ? nb[g] : 0;
  int s = w;  // columns up to and including this entry's
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += v;
  }
  const unsigned fit = __ballot_sync(0xffffffffu, in && s <= maxcol);
  const int take = __popc(fit);  // s does not decrease, so the entries that fit come first
  if (lane < take) {
    const int64_t t0 = off2[en.t] - tbase, c0 = offC[en.p3] + (int64_t)(onsite[en.p3] ? 0 : na[g]) * w * nbE;
    for (int k = 0; k < w; k++) {
      tb.t[s - w + k] = t0 + k;
      tb.c[s - w + k] = c0 + (int64_t)k * nbE;
      tb.nb[s - w + k] = w;
    }
  }
  if (lane == take - 1) {
    tb.n = s;
    tb.next = take;
  }
}

template <int R>
__global__ void __launch_bounds__(NT, R == 1 ? 4 : 1)
    k_X12(const int32_t *ord, const int64_t *ptr, const X12Entry *L, const int32_t *atomA2, const int32_t *atomB2,
          const int32_t *map2to1, const int32_t *map2to3, const int32_t *pA, const uint8_t *onsite, const int32_t *nb,
          const int32_t *na, const double *__restrict__ C, const int64_t *offC, const double *__restrict__ V,
          const int64_t *offV, const uint8_t *keepC, const uint8_t *keepV, const double *__restrict__ T,
          const int64_t *off2, const double *__restrict__ U, const int64_t *offU, const int64_t *offK, double *X,
          int64_t tbase, int smb, int t2, const uint8_t *t1tc, const uint8_t *rep1, const uint8_t *liveT, int ns) {
  extern __shared__ double sm[];
  __shared__ XCols tb;
  const int tid = threadIdx.x;
  const int s = ord[blockIdx.x / ns];
  const int rank = blockIdx.x % ns;
  const int a = atomA2[s], e = atomB2[s];
  const int nbA = nb[a], naA = na[a], nbE = nb[e], naE = na[e];
  const int nel = nbA * nbE;
  if ((R == 1) != (nel <= NT)) return;  // the other instance's output
  const int pae = map2to1[s];
  // term 1 in one orientation of each pair (rep1; else the transpose partner's block
  // carries it), and not for the column atoms whose term 1 runs on the tensor cores
  const bool has1 = pae >= 0 && keepV[pae] && rep1[pae] && !(t1tc && t1tc[e]);
  const double w1 = has1 && rep1[pae] == 2 ? 0.5 : 1.0;
  if (!has1 && !t2) return;
  const Split sp = split_of<R>(nel, rank, ns);
  double acc[R];
#pragma unroll
  for (int r = 0; r < R; r++) acc[r] = 0.0;
  if (has1) {
    const double *Vae = V + offV[pae];
    const int qlo = naE * rank / ns, qhi = naE * (rank + 1) / ns;  // this rank's Q on E'
    for (int64_t it = ptr[s]; it < ptr[s + 1];) {
      __syncthreads();
      if (tid < 32)
        x12_batch(tb, it, ptr[s + 1], min(XCOL, smb / nbA), L, keepC, pA, nb, na, onsite, off2, tbase, offC, nbE,
                  liveT);
      __syncthreads();
      const int n = tb.n;
      it += tb.next;
      if (n == 0) continue;
      const int per = nbA * n;
      const int qt = max(1, smb / per);
      for (int q0 = qlo; q0 < qhi; q0 += qt) {
        const int qn = min(qt, qhi - q0);
        if (q0 > qlo) __syncthreads();
        for (int el = tid; el < qn * per; el += NT) {
          const int q = el / per, rem = el - q * per;
          const int i = rem / n, c = rem - i * n;
          const int nbG = tb.nb[c];
          const double *tp = T + tb.t[c] + (int64_t)i * nbG;
          const double *vp = Vae + q0 + q;
          const int st = nbA * nbG;
          double u = 0.0;
#pragma unroll 4
          for (int P = 0; P < naA; P++) {
            u = fma(__ldg(vp), __ldg(tp), u);
            vp += naE;
            tp += st;
          }
          sm[el] = w1 * u;
        }
        __syncthreads();
        if (sp.grp < sp.ng) {
          const int K = qn * n;
          const int k0 = K * sp.grp / sp.ng, k1 = K * (sp.grp + 1) / sp.ng;
#pragma unroll
          for (int r = 0; r < R; r++) {
            const int el = sp.el0 + r * NT;
            if (el < nel) {
              const int i = el / nbE, l = el - i * nbE;
              int q = k0 / n, c = k0 - q * n;
              const double *up = sm + ((int64_t)q * nbA + i) * n + c;
              double v = 0.0;
#pragma unroll 4
              for (int k = k0; k < k1; k++) {
                v = fma(*up, __ldg(C + tb.c[c] + (int64_t)(q0 + q) * (tb.nb[c] * nbE) + l), v);
                up++;
                if (++c == n) {  // the next Q: same row i
                  c = 0;
                  q++;
                  up += (nbA - 1) * n;
                }
              }
              acc[r] += v;
            }
          }
        }
      }
    }
  }
  if (t2) {
    // term 2: X += U2(A,G')[Q][i][k] C(G',E')[Q on G'][k][l] (on the tensor cores in mixed precision)
    for (int64_t it = ptr[s]; it < ptr[s + 1]; it++) {
      const X12Entry en = L[it];
      if (en.u2 < 0 || !keepC[en.p3] || !keepV[en.u2] || (liveT && !liveT[en.t])) continue;
      const int g = pA[en.p3];
      dot_share<R>(acc, sp, nel, U + offU[en.u2], C + offC[en.p3], na[g], nbA, nb[g], nbE);
    }
  }
  double *out = X + offK[map2to3[s]];
  gather_shares<R>(acc, sp, nel, ns, sm, [&](int el, double v) { out[el] += v; });
}

// ------------------------------------------------------------------ term 4 intermediate
// Z(B,E')[P][j][l] = sum over (pair (B,G'), pair (G',E') not on-site) of
//   w sum_k D(B,G')[j][k] F[P][k][l],  F[P][k][l] = sum_Q V(B,G')[P][Q] C(G',E')[Q on G'][k][l],
// w the pair's weight (wZ: 1/2, or 1 for the pairs that stand for both orientations).
__global__ void __launch_bounds__(NT) k_Z(const int2 *items, const int64_t *ptrZ, const int2 *LZ,
                                          const int32_t *atomA2, const int32_t *atomB2, const int64_t *off2,
                                          const int32_t *pB, const int32_t *nb, const int32_t *na,
                                          const double *__restrict__ C, const int64_t *offC,
                                          const double *__restrict__ V, const int64_t *offV,
                                          const double *__restrict__ D, const int64_t *offD,
                                          const uint8_t *keepC, const uint8_t *keepV, const uint8_t *keepD,
                                          double *Z, int64_t zbase, int smb, const uint8_t *ztc,
                                          const uint8_t *wZ, int cap, PScreen ps) {
  extern __shared__ double sm[];
  const int tid = threadIdx.x;
  const int2 it = items[blockIdx.x];
  const int z = it.x, p0 = it.y;
  const int b = atomA2[z], e = atomB2[z];
  const int nbB = nb[b], naB = na[b], nbE = nb[e];
  const int per = nbB * nbE;
  const int pt = max(1, cap / per);
  const int pe = min(naB, p0 + pt);
  const int nel = (pe - p0) * per;
  double acc[MAXE];
#pragma unroll
  for (int r = 0; r < MAXE; r++) acc[r] = 0.0;
  for (int64_t x = ptrZ[z]; x < ptrZ[z + 1]; x++) {
    const int2 en = LZ[x];
    if (!keepD[en.x] || !keepV[en.x] || !keepC[en.y] || ps.drop3(en.x, en.x, en.y)) continue;
    const int g = pB[en.x];
    if (ztc && ztc[g]) continue;  // this middle atom's part runs on the tensor cores
    const int nbG = nb[g], naG = na[g];
    const double *Dbg = D + offD[en.x];
    const double *Vbg = V + offV[en.x];
    const double *Cge = C + offC[en.y];
    const double w = wZ[en.x] == 2 ? 0.5 : 1.0;
    const int fper = nbG * nbE;
    const int ft = max(1, min(pe - p0, smb / fper));
    for (int ps = p0; ps < pe; ps += ft) {
      const int fn = min(ft, pe - ps);
      __syncthreads();
      for (int el = tid; el < fn * fper; el += NT) {
        const int pp = el / fper, c = el - pp * fper;
        const double *vr = Vbg + (int64_t)(ps + pp) * naG;
        double f = 0.0;
        for (int Q = 0; Q < naG; Q++) f = fma(__ldg(vr + Q), __ldg(Cge + (int64_t)Q * fper + c), f);
        sm[el] = w * f;
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < MAXE; r++) {
        const int el = tid + r * NT;
        if (el < nel) {
          const int P = el / per;               // relative to p0
          const int pr = P - (ps - p0);
          if (pr >= 0 && pr < fn) {
            const int rem = el - P * per;
            const int j = rem / nbE, l = rem - j * nbE;
            const double *dj = Dbg + j * nbG;
            const double *fp = sm + pr * fper + l;
            double v = acc[r];
            for (int k = 0; k < nbG; k++) v = fma(__ldg(dj + k), fp[k * nbE], v);
            acc[r] = v;
          }
        }
      }
    }
  }
  double *out = Z + (off2[z] - zbase) + (int64_t)p0 * per;
#pragma unroll
  for (int r = 0; r < MAXE; r++) {
    const int el = tid + r * NT;
    if (el < nel) out[el] = acc[r];
  }
}

// ------------------------------------------------------------------ term 4 (and term 3 via the transpose)
// X(A,E') += sum over (C(A,B') not on-site, Z(B,E'')) of C(A,B')[P on B'][i][j] Z[P][j][l].
template <int R>
__global__ void __launch_bounds__(NT, R == 1 ? 6 : 1)
    k_X34(const int32_t *ord, const int64_t *ptr, const int2 *L, const int32_t *atomA3, const int32_t *atomB3,
          const int32_t *pB, const int32_t *nb, const int32_t *na, const double *__restrict__ C, const int64_t *offC,
          const uint8_t *keepC, const double *__restrict__ Z, const int64_t *off2, const int64_t *offK, double *X,
          int64_t zbase, int64_t zlo, int64_t zhi, const uint8_t *rep3, const uint8_t *liveZ, int ns) {
  __shared__ double red[R == 1 ? NT : NT * R];
  const int x = ord[blockIdx.x / ns];
  const int rank = blockIdx.x % ns;
  // term 4 halved in the K blocks: one orientation of each (the transpose partner carries
  // the other), with twice the weight of Z's 1/2; the self block keeps it.  Halved in Z
  // (rep3 = 2 everywhere): every block with weight 1.
  const uint8_t r3 = rep3[x];
  if (!r3) return;
  const double w4 = r3 == 2 ? 1.0 : 2.0;
  const int a = atomA3[x], e = atomB3[x];
  const int nbA = nb[a], naA = na[a], nbE = nb[e];
  const int nel = nbA * nbE;
  if ((R == 1) != (nel <= NT)) return;  // the other instance's output
  const Split sp = split_of<R>(nel, rank, ns);
  double acc[R];
#pragma unroll
  for (int r = 0; r < R; r++) acc[r] = 0.0;
  for (int64_t it = ptr[x]; it < ptr[x + 1]; it++) {
    const int2 en = L[it];
    if (!keepC[en.x] || en.y < zlo || en.y >= zhi || (liveZ && !liveZ[en.y])) continue;
    const int b = pB[en.x];
    const int nbB = nb[b];
    dot_share<R>(acc, sp, nel, C + offC[en.x] + (int64_t)naA * nbA * nbB, Z + (off2[en.y] - zbase), na[b], nbA, nbB,
                 nbE);
  }
  double *out = X + offK[x];
  gather_shares<R>(acc, sp, nel, ns, red, [&](int el, double v) { out[el] += w4 * v; });
}

// ------------------------------------------------------------------ K = X + X^T (image flipped)
// K(A,E,n) = X(A,E,n) + X(E,A,-n)^T (accumulate: added to K); a deterministic mixed
// build keeps the tensor-core part of X in 128-bit fixed point (X128) beside the FP64 part
__global__ void k_sym(int64_t nk, const int32_t *atomA3, const int32_t *atomB3, const int32_t *partner3,
                      const int32_t *nb, const int64_t *offK, const double *__restrict__ X,
                      const unsigned long long *X128, double *K, int accumulate) {
  const int64_t x = blockIdx.x;
  if (x >= nk) return;
  const int nbA = nb[atomA3[x]], nbE = nb[atomB3[x]];
  const int64_t oa = offK[x], ob = offK[partner3[x]];
  double *k = K + oa;
  for (int el = threadIdx.x; el < nbA * nbE; el += blockDim.x) {
    const int i = el / nbE, l = el - i * nbE;
    const int64_t ea = oa + el, eb = ob + l * nbA + i;
    double va = X[ea], vb = X[eb];
    if (X128) {
      va += from_x128(X128 + 2 * ea);
      vb += from_x128(X128 + 2 * eb);
    }
    const double v = va + vb;
    k[el] = accumulate ? k[el] + v : v;
  }
}

// ------------------------------------------------------------------ energy
// Pair p contributes sum_il D(B,A,-n)[l][i] K(A,B,n)[i][l].  A CTA takes 256 pairs, eight to a warp
// (lanes along the block's elements), and adds in a fixed tree.  (A thread per pair read both
// blocks element by element: 33 us for 576 pairs, 15 us now.)
constexpr int ENERGY_THREADS = 1024;
__global__ void __launch_bounds__(ENERGY_THREADS)
    k_energy(int64_t np, const int32_t *pA, const int32_t *pB, const int32_t *partner, const int32_t *map1to3,
             const int32_t *nb, const double *__restrict__ D, const int64_t *offD, const uint8_t *keepD,
             const double *__restrict__ K, const int64_t *offK, double *part) {
  __shared__ double red[ENERGY_THREADS / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = 0.0;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int64_t p = blockIdx.x * (int64_t)256 + warp + 32 * j;
    if (p >= np) continue;
    const int64_t q = partner[p];
    if (!keepD[q]) continue;
    const int nbA = nb[pA[p]], nbB = nb[pB[p]];
    const double *dq = D + offD[q];
    const double *kb = K + offK[map1to3[p]];
    for (int el = lane; el < nbA * nbB; el += 32) {
      const int i = el / nbB, l = el - i * nbB;
      s = fma(dq[l * nbA + i], kb[el], s);
    }
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  if (warp == 0) {
    s = red[lane];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) part[blockIdx.x] = s;
  }
}

// *Ex = scale * sum(part) (accumulate: *Ex += ...); scale -1/4 for the closed-shell energy
__global__ void k_energy_final(int64_t n, const double *part, double *Ex, double scale, int accumulate) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += 1024) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 512; w; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *Ex = accumulate ? *Ex + scale * red[0] : scale * red[0];
}

// ------------------------------------------------------------------ Gamma fold
__global__ void k_fold(int64_t ng, const int64_t *fold, const int32_t *atomA3, const int32_t *atomB3,
                       const int32_t *nb, const int64_t *offK, const int64_t *bofs, int64_t nbasis,
                       const double *__restrict__ K, double *Kd) {
  const int64_t gi = blockIdx.x;
  if (gi >= ng) return;
  const int64_t x0 = fold[gi], x1 = fold[gi + 1];
  const int a = atomA3[x0], e = atomB3[x0];
  const int nbA = nb[a], nbE = nb[e];
  for (int el = threadIdx.x; el < nbA * nbE; el += blockDim.x) {
    double s = 0.0;
    for (int64_t x = x0; x < x1; x++) s += K[offK[x] + el];
    const int i = el / nbE, l = el - i * nbE;
    Kd[(bofs[a] + i) * nbasis + bofs[e] + l] = s;
  }
}

rix_status fail_cuda(rix_ctx *ctx, const char *what, cudaError_t e) {
  ctx->last_error = std::string(what) + ": " + cudaGetErrorString(e);
  return RIX_ECUDA;
}

rix_status last(rix_ctx *ctx, const char *what) {
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RIX_OK : fail_cuda(ctx, what, e);
}

}  // namespace

rix_status rix_launch_pairs(rix_ctx *ctx, const double *d_xyz, const double *d_cell, const int nr[3],
                            int64_t *d_counts, const int64_t *d_rowptr, int64_t *d_keys, cudaStream_t st) {
  const int nat = ctx->nat;
  const int threads = 256;
  const int64_t blocks = ((int64_t)nat * 32 + threads - 1) / threads;
  k_pairs<<<(unsigned)blocks, threads, 0, st>>>(nat, d_xyz, d_cell, ctx->periodic ? 1 : 0, nr[0], nr[1], nr[2],
                                                ctx->rc * ctx->rc, ctx->rc > 0 ? 1 : 0, d_counts, d_rowptr, d_keys);
  return last(ctx, "k_pairs");
}

rix_status rix_launch_flags(rix_ctx *ctx, const double *arr, const int64_t *off, int64_t n, uint8_t *keep,
                            cudaStream_t st, float *norm) {
  if (n == 0) return RIX_OK;
  float *nm = ctx->opt.product_tau > 0 ? norm : nullptr;
  if (off == ctx->d_offD) k_flags<1><<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>(arr, off, n, ctx->tau, keep, nm);
  else k_flags<8><<<(unsigned)n, 256, 0, st>>>(arr, off, n, ctx->tau, keep, nm);
  return last(ctx, "k_flags");
}

// out[a] = max over the pairs (a, .) of norm (one thread per atom)
__global__ void k_atom_max(int nat, const int64_t *row1, const float *norm, float *out) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nat) return;
  float m = 0.f;
  for (int64_t p = row1[a]; p < row1[a + 1]; p++) m = fmaxf(m, norm[p]);
  out[a] = m;
}

rix_status rix_launch_atom_max(rix_ctx *ctx, const float *norm, float *out, cudaStream_t st) {
  k_atom_max<<<(ctx->nat + 127) / 128, 128, 0, st>>>(ctx->nat, ctx->d_row1, norm, out);
  return last(ctx, "k_atom_max");
}

rix_status rix_launch_symcheck(rix_ctx *ctx, cudaStream_t st) {
  RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int32_t), st));
  k_symcheck<<<(unsigned)ctx->np, 256, 0, st>>>(ctx->d_pA, ctx->d_pB, ctx->d_partner1, ctx->d_onsite, ctx->d_nb,
                                                ctx->d_na, ctx->d_C, ctx->d_offC, ctx->d_V, ctx->d_offV, ctx->d_flag);
  return last(ctx, "k_symcheck");
}

// Shared memory up to SM_MAX doubles for the kernels that stage tiles, and clusters of 16 CTAs, which
// are beyond the portable size.  Set for every context, on its device.
rix_status rix_fp64_attrs(rix_ctx *ctx) {
  auto set = [&](auto *kernel, int smem, bool cluster) {
    cudaError_t e = cudaSuccess;
    if (smem) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess && cluster) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  };
  RIX_CUDA_TRY(ctx, set(k_X12<1>, SM_MAX * 8, true));
  RIX_CUDA_TRY(ctx, set(k_X12<XMAXE>, SM_MAX * 8, true));
  RIX_CUDA_TRY(ctx, set(k_X34<1>, 0, true));
  RIX_CUDA_TRY(ctx, set(k_X34<XMAXE>, 0, true));
  RIX_CUDA_TRY(ctx, set(k_T, TCOL * 64 * 8, false));
  RIX_CUDA_TRY(ctx, set(k_Z, SM_MAX * 8, false));
  return RIX_OK;
}

namespace {

// the configuration of count outputs, each shared by a cluster of ns CTAs (at: its attribute)
cudaLaunchConfig_t split_config(int64_t count, int ns, int smem, cudaStream_t st, cudaLaunchAttribute *at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * ns));
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = ns;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = ns > 1 ? 1 : 0;
  return cfg;
}

// whether the device (or the part of it that the context has) runs clusters of ns CTAs of the kernel
template <class... P>
bool cluster_fits(void (*kernel)(P...), int ns, int smem) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = split_config(1, ns, smem, 0, &at);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess) return n > 0;
  cudaGetLastError();
  return false;
}

}  // namespace

int rix_cluster_limit(int want) {
  return fitting_class(want, [](int ns) {  // k_X12 with the largest tile that the autotuner may choose
    return cluster_fits(k_X12<1>, ns, SM_MAX * 8) && cluster_fits(k_X12<XMAXE>, ns, SM_MAX * 8) &&
           cluster_fits(k_X34<1>, ns, 0) && cluster_fits(k_X34<XMAXE>, ns, 0);
  });
}

namespace {

// Z(B;E') for the Z work items [first, first + count) of block b.
rix_status launch_Z_items(rix_ctx *ctx, const double *D, int b, int64_t first, int64_t count, int smb,
                          cudaStream_t st) {
  if (!count) return RIX_OK;
  smb = std::max(smb, ctx->max_nel);  // one row of F, nbG x nbE: a cached budget may be smaller
  k_Z<<<(unsigned)count, NT, smb * 8, st>>>(ctx->d_itZ + ctx->segZ[b] + first, ctx->d_ptrZ, ctx->d_LZ,
                                            ctx->d_atomA2, ctx->d_atomB2, ctx->d_off2, ctx->d_pB, ctx->d_nb,
                                            ctx->d_na, ctx->d_C, ctx->d_offC, ctx->d_V, ctx->d_offV, D, ctx->d_offD,
                                            ctx->d_keepC, ctx->d_keepV, ctx->d_keepD, ctx->d_Z, ctx->blk_base[b],
                                            smb, ctx->have_mx ? ctx->d_ztc : nullptr, ctx->d_wZ, ctx->cap_Z,
                                            rix_pscreen(ctx));
  return last(ctx, "k_Z");
}

// a launch of count outputs, each shared by a cluster of ns CTAs
template <class... P, class... A>
cudaError_t launch_split(void (*kernel)(P...), int64_t count, int ns, int smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = split_config(count, ns, smem, st, &at);
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// the live flags of the T and Z blocks for the current D flags
rix_status launch_live(rix_ctx *ctx, cudaStream_t st) {
  if (!ctx->use_live) return RIX_OK;
  const unsigned grid = (unsigned)((ctx->n2 * 32 + 255) / 256);
  k_live<<<grid, 256, 0, st>>>(ctx->n2, ctx->d_ptrT, ctx->d_LT, ctx->d_keepC, nullptr, ctx->d_keepD, rix_pscreen(ctx),
                               ctx->d_live2);
  k_live<<<grid, 256, 0, st>>>(ctx->n2, ctx->d_ptrZ, ctx->d_LZ, ctx->d_keepC, ctx->d_keepV, ctx->d_keepD,
                               rix_pscreen(ctx), ctx->d_live2 + ctx->n2);
  return last(ctx, "k_live");
}

// outputs of terms 1+2 in block b
int64_t n_X12(const rix_ctx *ctx, int b) {
  return ctx->segX12[rix_ctx::NCLS * (b + 1)] - ctx->segX12[rix_ctx::NCLS * b];
}

// terms 1+2 for the output blocks [first, first + count) of block b's launch order.
rix_status launch_X12_items(rix_ctx *ctx, int b, int64_t first, int64_t count, int smb, cudaStream_t st) {
  smb = std::max(smb, 64 * 64);  // one column entry of 64 functions over 64 rows, or a 64 x 64 output
  const int64_t *seg = &ctx->segX12[rix_ctx::NCLS * b];
  for (int c = 0; c < rix_ctx::NCLS; c++) {  // the class's part of [first, first + count)
    const int64_t lo = std::max(seg[c], seg[0] + first), hi = std::min(seg[c + 1], seg[0] + first + count);
    if (hi <= lo) continue;
    auto go = [&](auto *kernel) {
      return launch_split(kernel, hi - lo, 1 << c, smb * 8, st, ctx->d_ordX12 + lo, ctx->d_ptrX12, ctx->d_LX12,
                          ctx->d_atomA2, ctx->d_atomB2, ctx->d_map2to1, ctx->d_map2to3, ctx->d_pA, ctx->d_onsite,
                          ctx->d_nb, ctx->d_na, ctx->d_C, ctx->d_offC, ctx->d_V, ctx->d_offV, ctx->d_keepC,
                          ctx->d_keepV, ctx->d_T, ctx->d_off2, ctx->d_U, ctx->d_offU, ctx->d_offK, ctx->d_X,
                          ctx->blk_base[b], smb, ctx->have_mx ? 0 : 1, ctx->have_mx ? ctx->d_t1tc : nullptr,
                          ctx->d_rep1, ctx->use_live ? ctx->d_live2 : nullptr, 1 << c);
    };
    cudaError_t e = go(k_X12<1>);
    if (e == cudaSuccess && ctx->max_nel > NT) e = go(k_X12<XMAXE>);
    if (e != cudaSuccess) return fail_cuda(ctx, "k_X12", e);
  }
  return last(ctx, "k_X12");
}

// terms 3+4 (FP64) for every K block, Z of block b.
rix_status launch_X34(rix_ctx *ctx, int b, cudaStream_t st) {
  const int64_t zlo = ctx->row2[ctx->blk_atom[b]], zhi = ctx->row2[ctx->blk_atom[b + 1]];
  for (int c = 0; c < rix_ctx::NCLS; c++) {
    const int64_t lo = ctx->segX34[c], n = ctx->segX34[c + 1] - lo;
    if (!n) continue;
    auto go = [&](auto *kernel) {
      return launch_split(kernel, n, 1 << c, 0, st, ctx->d_ordX34 + lo, ctx->d_ptrX34, ctx->d_LX34, ctx->d_atomA3,
                          ctx->d_atomB3, ctx->d_pB, ctx->d_nb, ctx->d_na, ctx->d_C, ctx->d_offC, ctx->d_keepC,
                          ctx->d_Z, ctx->d_off2, ctx->d_offK, ctx->d_X, ctx->blk_base[b], zlo, zhi, ctx->d_rep3,
                          ctx->use_live ? ctx->d_live2 + ctx->n2 : nullptr, 1 << c);
    };
    cudaError_t e = go(k_X34<1>);
    if (e == cudaSuccess && ctx->max_nel > NT) e = go(k_X34<XMAXE>);
    if (e != cudaSuccess) return fail_cuda(ctx, "k_X34", e);
  }
  return last(ctx, "k_X34");
}

}  // namespace

// one launch per class that has outputs, and a second one for the K blocks above 256 elements
int32_t rix_x12_launches(const rix_ctx *ctx) {
  int32_t n = 0;
  for (size_t i = 0; i + 1 < ctx->segX12.size(); i++) n += ctx->segX12[i + 1] > ctx->segX12[i];
  return ctx->max_nel > NT ? 2 * n : n;
}

int32_t rix_x34_launches(const rix_ctx *ctx) {
  int32_t n = 0;
  for (int c = 0; c < rix_ctx::NCLS; c++) n += ctx->segX34[c + 1] > ctx->segX34[c];
  return ctx->max_nel > NT ? 2 * n : n;
}

// T(A,G') for the row atoms of block b (T buffer holds that block).  In mixed
// precision the buffer is cleared first and the tensor cores add the T blocks
// of their row atoms; k_T stores the others, if there are any ((H2O)8, all on the tensor cores:
// a launch of CTAs that return at once took 11 of 1,390 us).
rix_status rix_launch_T_block(rix_ctx *ctx, const double *D, int b, cudaStream_t st) {
  const int64_t nT = ctx->segT[b + 1] - ctx->segT[b];
  const bool tc = ctx->have_mx && ctx->n_ttc > 0;
  if (tc) {
    const int64_t n = ctx->off2[ctx->row2[ctx->blk_atom[b + 1]]] - ctx->blk_base[b];
    RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_T, 0, sizeof(double) * n, st));
  }
  if (nT && !(tc && ctx->n_ttc == ctx->nat)) {
    k_T<<<(unsigned)nT, NT, TCOL * ctx->max_nb * 8, st>>>(ctx->d_itT + ctx->segT[b], ctx->d_ptrT, ctx->d_LT, ctx->d_atomA2,
                                               ctx->d_atomB2, ctx->d_off2, ctx->d_pB, ctx->d_nb, ctx->d_na,
                                               ctx->d_C, ctx->d_offC, D, ctx->d_offD, ctx->d_keepC, ctx->d_keepD,
                                               ctx->d_T, ctx->blk_base[b], tc ? ctx->d_ttc : nullptr, ctx->cap_T,
                                               rix_pscreen(ctx));
    rix_status s = last(ctx, "k_T");
    if (s != RIX_OK) return s;
  }
  return tc ? rix_mixed_T(ctx, b, ctx->blk_base[b], D, st) : RIX_OK;
}

// Z(B;E') for the middle atoms of block b (Z buffer holds that block): the FP64
// kernel stores its part, then in mixed precision the tensor cores add theirs.
rix_status rix_launch_Z_block(rix_ctx *ctx, const double *D, int b, cudaStream_t st) {
  rix_status s = RIX_OK;
  if (ctx->have_mx && ctx->n_ztc == ctx->nat) {
    // every middle atom runs on the tensor cores: the FP64 kernel would only write zeros
    const int64_t n = ctx->off2[ctx->row2[ctx->blk_atom[b + 1]]] - ctx->blk_base[b];
    RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_Z, 0, sizeof(double) * n, st));
  } else {
    s = launch_Z_items(ctx, D, b, 0, ctx->segZ[b + 1] - ctx->segZ[b], ctx->tile_Z, st);
  }
  if (s == RIX_OK && ctx->have_mx) s = rix_mixed_z(ctx, b, ctx->blk_base[b], D, st);
  return s;
}

rix_status rix_fp64_build(rix_ctx *ctx, const double *D, double *K, cudaStream_t st, int accumulate) {
  rix_status s;
  if ((s = rix_prof_mark(ctx, 0, st)) != RIX_OK) return s;
  if ((s = rix_launch_flags(ctx, D, ctx->d_offD, ctx->np, ctx->d_keepD, st, ctx->d_normD)) != RIX_OK) return s;
  if ((s = launch_live(ctx, st)) != RIX_OK) return s;
  if ((s = rix_prof_mark(ctx, 1, st)) != RIX_OK) return s;
  RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_X, 0, sizeof(double) * ctx->offK[ctx->nk], st));
  if (ctx->d_X128)
    RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_X128, 0, 2 * sizeof(unsigned long long) * ctx->offK[ctx->nk], st));
  // terms 1 and 2, one block of row atoms at a time (T resident for the block)
  for (int b = 0; b < ctx->nblk; b++) {
    const int64_t tbase = ctx->blk_base[b];
    if ((s = rix_launch_T_block(ctx, D, b, st)) != RIX_OK) return s;
    if (b == 0 && (s = rix_prof_mark(ctx, 2, st)) != RIX_OK) return s;
    const int64_t nU = ctx->segU[b + 1] - ctx->segU[b];
    if (nU) {
      k_U2<<<(unsigned)nU, NT, 0, st>>>(ctx->d_itU + ctx->segU[b], ctx->d_pA, ctx->d_pB, ctx->d_nb, ctx->d_na,
                                        ctx->d_V, ctx->d_offV, ctx->d_keepV, ctx->d_map1to2, ctx->d_T, ctx->d_off2,
                                        ctx->d_offU, ctx->d_U, tbase, ctx->cap_U);
      if ((s = last(ctx, "k_U2")) != RIX_OK) return s;
    }
    if (b == 0 && (s = rix_prof_mark(ctx, 3, st)) != RIX_OK) return s;
    if ((!ctx->have_mx || ctx->n_t1tc < ctx->nat) &&
        (s = launch_X12_items(ctx, b, 0, n_X12(ctx, b), ctx->tile_X12, st)) != RIX_OK)
      return s;
    // mixed precision, several row blocks: term 1 on the tensor cores while T of the block is resident
    if (ctx->have_mx && ctx->nblk > 1 && (s = rix_mixed_t1(ctx, b, tbase, st)) != RIX_OK) return s;
  }
  if ((s = rix_prof_mark(ctx, 4, st)) != RIX_OK) return s;
  // mixed precision: term 1 (single block) and term 2 on the tensor cores
  if (ctx->have_mx && ctx->nblk == 1 && (s = rix_mixed_t1(ctx, 0, ctx->blk_base[0], st)) != RIX_OK) return s;
  if (ctx->have_mx && (s = rix_mixed_t2(ctx, st)) != RIX_OK) return s;
  if ((s = rix_prof_mark(ctx, 5, st)) != RIX_OK) return s;
  // terms 3 and 4, one block of middle atoms B at a time (Z resident for the block)
  for (int b = 0; b < ctx->nblk; b++) {
    const int64_t zbase = ctx->blk_base[b];
    if ((s = rix_launch_Z_block(ctx, D, b, st)) != RIX_OK) return s;
    if (b == 0 && (s = rix_prof_mark(ctx, 6, st)) != RIX_OK) return s;
    if (ctx->have_mx) {
      if ((s = rix_mixed_x34(ctx, b, zbase, st)) != RIX_OK) return s;
    } else if ((s = launch_X34(ctx, b, st)) != RIX_OK) {
      return s;
    }
  }
  if ((s = rix_prof_mark(ctx, 7, st)) != RIX_OK) return s;
  k_sym<<<(unsigned)ctx->nk, 128, 0, st>>>(ctx->nk, ctx->d_atomA3, ctx->d_atomB3, ctx->d_partner3, ctx->d_nb,
                                           ctx->d_offK, ctx->d_X, ctx->d_X128, K, accumulate);
  if ((s = last(ctx, "k_sym")) != RIX_OK) return s;
  return rix_prof_mark(ctx, 8, st);
}

// ------------------------------------------------------------------ autotuner
// Picks the shared-memory tile budget of k_X12 and k_Z (and with it their
// tile shapes and CTAs per SM; k_X34 stages nothing and keeps its entry) by timing each candidate on a slice of
// the real work items of the first memory-plan block; the choice is cached
// per system in a text file.  The analogue of the paper's auto-tuned Fock
// block size (Sec. "Initialization"), at the level of one GPU's tiles.
namespace {

constexpr int N_CAND = 4;
constexpr int CAND[N_CAND] = {4096, 8192, 12288, 16384};

std::string tune_key(const rix_ctx *ctx) {
  cudaDeviceProp prop;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaGetDeviceProperties(&prop, dev);
  char buf[512];
  // k2: the kernels the tiles were timed with; a choice made for others (96 KB a CTA, where k_X12
  // now takes 32 KB) is not theirs
  snprintf(buf, sizeof buf, "%s|k2|nat=%d|np=%lld|n2=%lld|nk=%lld|prec=%d|blk=%d|", prop.name, ctx->nat,
           (long long)ctx->np, (long long)ctx->n2, (long long)ctx->nk, (int)ctx->opt.precision, ctx->nblk);
  std::string k(buf);
  for (char &c : k)
    if (c == ' ') c = '_';
  return k;
}

// time `launch(c)` for every candidate c (one untimed run first); returns the fastest
template <class F>
rix_status pick(rix_ctx *ctx, cudaStream_t st, F launch, int *best, float *best_ms) {
  cudaEvent_t e0, e1;
  RIX_CUDA_TRY(ctx, cudaEventCreate(&e0));
  RIX_CUDA_TRY(ctx, cudaEventCreate(&e1));
  *best_ms = 3.0e38f;
  rix_status s = RIX_OK;
  for (int c = 0; c < N_CAND && s == RIX_OK; c++) {
    if ((s = launch(CAND[c])) != RIX_OK) break;
    cudaEventRecord(e0, st);
    if ((s = launch(CAND[c])) != RIX_OK) break;
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess) { s = RIX_ECUDA; break; }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < *best_ms) { *best_ms = ms; *best = CAND[c]; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return s;
}

}  // namespace

extern "C" rix_status rix_autotune(rix_ctx *ctx, const double *D, const char *cache_path, int32_t *chosen,
                                   void *stream) {
  if (!ctx || !D) return RIX_EINVAL;
  if (!ctx->have_cv) return RIX_ESTATE;
  cudaStream_t st = (cudaStream_t)stream;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (st && cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
    ctx->last_error = "rix_autotune times kernels and cannot run inside a graph capture";
    return RIX_ESTATE;
  }
  ctx->fwd_valid = false;  // the timing runs overwrite the intermediates
  const std::string key = tune_key(ctx);
  if (cache_path && *cache_path) {
    if (FILE *f = fopen(cache_path, "r")) {
      char line[1024];
      while (fgets(line, sizeof line, f)) {
        char k[600];
        int a = 0, b = 0, c = 0;
        if (sscanf(line, "%599s %d %d %d", k, &a, &b, &c) == 4 && key == k && a > 0 && b > 0 && c > 0 &&
            a <= SM_MAX && b <= SM_MAX && c <= SM_MAX) {
          ctx->tile_X12 = a, ctx->tile_Z = b, ctx->tile_X34 = c;
          fclose(f);
          if (chosen) chosen[0] = a, chosen[1] = b, chosen[2] = c;
          return RIX_OK;
        }
      }
      fclose(f);
    }
  }
  rix_status s;
  if ((s = rix_launch_flags(ctx, D, ctx->d_offD, ctx->np, ctx->d_keepD, st)) != RIX_OK) return s;
  if ((s = launch_live(ctx, st)) != RIX_OK) return s;
  RIX_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_X, 0, sizeof(double) * ctx->offK[ctx->nk], st));
  const int b = 0;
  const int64_t SAMPLE = 4096;
  // block 0's T and U2 feed the term 1+2 sample
  if ((s = rix_launch_T_block(ctx, D, b, st)) != RIX_OK) return s;
  const int64_t nU = ctx->segU[b + 1] - ctx->segU[b];
  if (nU) {
    k_U2<<<(unsigned)nU, NT, 0, st>>>(ctx->d_itU + ctx->segU[b], ctx->d_pA, ctx->d_pB, ctx->d_nb, ctx->d_na,
                                      ctx->d_V, ctx->d_offV, ctx->d_keepV, ctx->d_map1to2, ctx->d_T, ctx->d_off2,
                                      ctx->d_offU, ctx->d_U, ctx->blk_base[b], ctx->cap_U);
    if ((s = last(ctx, "k_U2")) != RIX_OK) return s;
  }
  float ms = 0.f;
  {
    const int64_t n = n_X12(ctx, b), cnt = std::min(n, SAMPLE), first = (n - cnt) / 2;
    if (cnt && (s = pick(ctx, st, [&](int c) { return launch_X12_items(ctx, b, first, cnt, c, st); },
                         &ctx->tile_X12, &ms)) != RIX_OK)
      return s;
  }
  {
    const int64_t n = ctx->segZ[b + 1] - ctx->segZ[b], cnt = std::min(n, SAMPLE), first = (n - cnt) / 2;
    if (cnt && (s = pick(ctx, st, [&](int c) { return launch_Z_items(ctx, D, b, first, cnt, c, st); },
                         &ctx->tile_Z, &ms)) != RIX_OK)
      return s;
  }
  RIX_CUDA_TRY(ctx, cudaStreamSynchronize(st));
  if (cache_path && *cache_path) {
    if (FILE *f = fopen(cache_path, "a")) {
      fprintf(f, "%s %d %d %d\n", key.c_str(), ctx->tile_X12, ctx->tile_Z, ctx->tile_X34);
      fclose(f);
    }
  }
  if (chosen) chosen[0] = ctx->tile_X12, chosen[1] = ctx->tile_Z, chosen[2] = ctx->tile_X34;
  return RIX_OK;
}

rix_status rix_launch_energy(rix_ctx *ctx, const double *D, const double *K, double *Ex, cudaStream_t st) {
  rix_status s;
  if ((s = rix_launch_flags(ctx, D, ctx->d_offD, ctx->np, ctx->d_keepD, st)) != RIX_OK) return s;
  k_energy<<<(unsigned)ctx->n_epart, ENERGY_THREADS, 0, st>>>(ctx->np, ctx->d_pA, ctx->d_pB, ctx->d_partner1, ctx->d_map1to3,
                                                   ctx->d_nb, D, ctx->d_offD, ctx->d_keepD, K, ctx->d_offK,
                                                   ctx->d_epart);
  if ((s = last(ctx, "k_energy")) != RIX_OK) return s;
  k_energy_final<<<1, 1024, 0, st>>>(ctx->n_epart, ctx->d_epart, Ex, -0.25, 0);
  return last(ctx, "k_energy_final");
}

// scale * sum over the D pattern of <D(E,A,-n), K(A,E,n)> into (or added to) *Ex
rix_status rix_launch_energy_scaled(rix_ctx *ctx, const double *D, const double *K, double *Ex, double scale,
                                    int accumulate, cudaStream_t st) {
  rix_status s;
  if ((s = rix_launch_flags(ctx, D, ctx->d_offD, ctx->np, ctx->d_keepD, st)) != RIX_OK) return s;
  k_energy<<<(unsigned)ctx->n_epart, ENERGY_THREADS, 0, st>>>(ctx->np, ctx->d_pA, ctx->d_pB, ctx->d_partner1, ctx->d_map1to3,
                                                   ctx->d_nb, D, ctx->d_offD, ctx->d_keepD, K, ctx->d_offK,
                                                   ctx->d_epart);
  if ((s = last(ctx, "k_energy")) != RIX_OK) return s;
  k_energy_final<<<1, 1024, 0, st>>>(ctx->n_epart, ctx->d_epart, Ex, scale, accumulate);
  return last(ctx, "k_energy_final");
}

// Same energy reduction as rix_launch_energy, with the per-CTA partial sums in
// a caller-supplied device buffer of at least ctx->n_epart doubles.
rix_status rix_launch_energy_partials(rix_ctx *ctx, const double *D, const double *K, double *Ex, double *partials,
                                      cudaStream_t st) {
  rix_status s;
  if ((s = rix_launch_flags(ctx, D, ctx->d_offD, ctx->np, ctx->d_keepD, st)) != RIX_OK) return s;
  k_energy<<<(unsigned)ctx->n_epart, ENERGY_THREADS, 0, st>>>(ctx->np, ctx->d_pA, ctx->d_pB, ctx->d_partner1, ctx->d_map1to3,
                                                   ctx->d_nb, D, ctx->d_offD, ctx->d_keepD, K, ctx->d_offK,
                                                   partials);
  if ((s = last(ctx, "k_energy")) != RIX_OK) return s;
  k_energy_final<<<1, 1024, 0, st>>>(ctx->n_epart, partials, Ex, -0.25, 0);
  return last(ctx, "k_energy_final");
}

rix_status rix_launch_fold(rix_ctx *ctx, const double *K, double *Kd, cudaStream_t st) {
  RIX_CUDA_TRY(ctx, cudaMemsetAsync(Kd, 0, sizeof(double) * ctx->nbasis * ctx->nbasis, st));
  k_fold<<<(unsigned)ctx->n_fold, 128, 0, st>>>(ctx->n_fold, ctx->d_fold, ctx->d_atomA3, ctx->d_atomB3, ctx->d_nb,
                                                ctx->d_offK, ctx->d_bofs, ctx->nbasis, K, Kd);
  return last(ctx, "k_fold");
}
