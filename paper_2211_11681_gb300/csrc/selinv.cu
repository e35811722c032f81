// Selected inversion on the compression pattern (Sec. 4.2 "Sparse selected inversion",
// Eq. (blockInv)) and the contour-integral inverse square root (Sec. 4.4, Eq. (ContInt)),
// in FP64.
//
// Supernodes are the clusters: every non-empty cluster is one block column of the factor,
// its samplets a dense block.  The host picks a minimum-degree elimination order of the
// block graph of S, plays the elimination game to get the pattern of L (position space,
// i >= k), and lists the blocks of every level of the elimination tree.  Blocks whose
// columns sit on one level are independent, so each level is one launch per step:
//
//   factor, levels from the leaves up (A + sigma I = L D L^T, W = L D kept beside L):
//     update  W(i,k) = A(i,k) + sigma [i = k] - sum_{j < k} W(i,j) L(k,j)^T over the j in
//             both row i and row k of L;
//     pivot   D(k,k) = W(k,k) inverted by Gauss-Jordan in shared memory (positive definite:
//             no pivoting; a pivot that is not positive is recorded), then
//             L(i,k) = W(i,k) D(k,k)^{-1} for the rows of column k (a CTA per supernode
//             and range of rows), D^{-1} stored in L's diagonal block;
//   inversion, levels from the root down (Takahashi-type recurrences from Eq. (blockInv)):
//     off     Z(i,k) = - sum_{j in struct(k)} Z(i,j) L(j,k), Z(i,j) read from block
//             (max, min) of Z, transposed when i < j;
//     diag    Z(k,k) = D(k,k)^{-1} - sum_{j in struct(k)} Z(j,k)^T L(j,k) (a CTA or a cluster of
//             CTAs per supernode, its warps splitting the sum);
//   scatter   out = alpha P_S(Z) + beta out, blocks of S read from Z or its transpose.
//
// The terms of every sum are fixed by the pattern of L, so the plan lists them once (the
// symbolic phase of both sweeps): per block of L the pairs (W(i,j), L(k,j)) of the update and
// (Z(i,j), L(j,k)) of the inversion.  A warp sums a tile of at most 20 x 20 entries of one output
// block over a part of its list, 8, 4 or 2 terms at a time dealt to its lanes as in the double
// product (si_sum): the FP64 pipe takes as long for 1 lane as for 32.  Near the root the
// elimination tree is a chain whose levels hold few, long sums, so the host splits each list
// over the 4 warps of a CTA and, where that leaves SMs idle, over several CTAs (split-K): the
// warps' sums are added in the CTA, the CTAs' parts land in a scratch buffer and the next
// launch of the level (pivot, diag) adds them, all in a fixed order, so results do not depend
// on scheduling.  What bounds a level is its chain of latencies (term list, operand offsets, copies,
// at least 8 terms' FP64 instructions) more than its operations; see the kernels.
//
// The launches overlap: each kernel starts while the one before it drains and fetches its first term
// lists and offsets (plan data) before it waits for that one's results.  At N = 8192 in the plane
// a factorization and an inversion are 1288 launches: 53.9 ms, 56.3 with launches in a row.
//
// Measured, factorization and inversion in the plane, 10-wide blocks (in brackets one entry per lane
// and term, sums split for sixteen warps a scheduler): N = 4096 22.7 ms (37.7), N = 8192 53.9 ms
// (82.8), N = 16384 172 ms (228), N = 65536 1.50 s (1.88), 0.75 TFLOP/s.
//
// Every entry a launch reads was written by an earlier launch (descendants sit on lower
// levels, ancestors on higher ones) or by its own CTA before a barrier, so the kernels need
// no synchronisation beyond that.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"
#include "sselinv.h"

namespace sf {
namespace {

constexpr int kSiMaxB = 64;               // widest block
constexpr int kSiWarps = 4;               // warps per CTA of the sum kernels
constexpr int kSiThreads = 256;           // threads of the pivot kernel
constexpr int kSiSlots = 25;              // accumulators of a lane
constexpr int kSiChains = 2;              // accumulators a full step works on at a time
constexpr int kSiBuf = 1600;              // doubles of a warp's stage buffer
constexpr int kSiChunk = 2048;            // doubles of W a pivot CTA holds at a time
constexpr int kSiCluster = 8;             // CTAs that share a long diagonal sum
constexpr int kSiStepTerms = 2;           // fewest terms worth a warp
constexpr int kSiMaxParts = 16;           // CTAs of one split sum
constexpr int kSiMaxClusters = 32768;     // non-empty clusters of the host bitset analysis

struct SiItem {
  int32_t blk;      // CSC block of L
  int32_t col;      // its column position
  int16_t r0, c0;   // tile of at most kTile x kTile entries
};

struct SiDev {
  const int32_t* bs;      // block size per position
  const int64_t* colptr;  // CSC of L: column k holds blocks colptr[k] .. colptr[k+1]-1,
  const int32_t* colrow;  //   the diagonal first, then the rows of struct(k) ascending
  const int64_t* loff;    // entry offset of each CSC block (rows x cols, row-major)
  const int64_t* lpo;     // entry offset of each CSC block among the blocks of its level
  const int32_t* colcol;  // column position of each CSC block
  const int64_t* uptr;    // factor terms of CSC block q: uptr[q] .. uptr[q+1]-1, pairs of
  const int32_t* uw;      //   CSC blocks W(i,j), L(k,j)
  const int32_t* ul;
  const int64_t* optr;    // inversion terms of CSC block q = (i,k), i > k: for every j in
  const int32_t* oz;      //   struct(k) the block of Z(i,j) (~index: stored as Z(j,i)) and
  const int32_t* ol;      //   the block L(j,k)
  const int64_t* aoff;    // per CSC block: entry offset of the S block with its rows and
                          // columns (-1: not in S)
  double* W;              // L D (D in the diagonal blocks)
  double* L;              // L (D^{-1} in the diagonal blocks)
  double* Z;              // the inverse on the pattern of L
  double* P;              // partial sums of split launches: [part][entries of the level]
  unsigned int* flag;     // mapped host word: 1 = a pivot block was not positive definite
};

// Which terms a sum runs over: the update's list, the inversion's list, or the blocks of column k.
enum { kSiUpdate, kSiOff, kSiDiag };

// One warp's sum over terms t .. te-1 (t steps of S) of a th x tw tile: sum of x(r0 + r, :) y(:, c0 + c).
// On return base[e] (e = r tw + c) holds the sum.  The operands of S terms are staged together
// and their (term, entry) pairs dealt to the lanes, kSiSlots accumulators each (the rules of
// mul_f64_kernel).  Blocks are staged in the order they are stored; the next terms' offsets are
// fetched while the copies arrive.
template <int MODE>
__device__ __forceinline__ void si_sum(const SiDev& s, int64_t t, int64_t te, int64_t q0, int bi, int bk, int r0, int c0,
                                       int th, int tw, double* base, int lane) {
  constexpr bool kYRows = MODE == kSiUpdate;  // y stored [c][t] (L(k,j)), else [t][c] (L(j,k))
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(base);
  const int ne = th * tw;
  const int S = ne <= 100 && th + tw <= 20 ? 8 : ne <= 200 ? 4 : 2;
  const int KC = S == 2 ? 20 : 10;
  double acc[kSiSlots];
  int off[kSiSlots];  // slot m: term s of the step, entry (r, c): s << 16 | r << 8 | c
  const float rne = 1.0f / (float)ne, rtw = 1.0f / (float)tw;
  const int used = (int)max((int64_t)0, min((int64_t)S, te - t)) * ne;  // (term, entry) pairs of a step at most
#pragma unroll
  for (int m = 0; m < kSiSlots; ++m) {
    acc[m] = 0.0;
    off[m] = 0;
    if (32 * m >= used) continue;
    const int i = min(lane + 32 * m, used - 1);
    const int u = __float2int_rz(((float)i + 0.5f) * rne), e = i - u * ne;
    const int r = __float2int_rz(((float)e + 0.5f) * rtw);
    off[m] = u << 16 | r << 8 | (e - r * tw);
  }
  // lane u holds term u of the next step: t extent (0: none; negative: x is stored transposed) and
  // where its operands start
  int nj = 0;
  int64_t nx = 0, ny = 0;
  auto fetch = [&](int64_t from) {
    nj = 0;
    const int64_t q = from + lane;
    if (lane >= S || q >= te) return;
    if (MODE == kSiUpdate) {
      const int bw = s.uw[q];
      nj = s.bs[s.colcol[bw]];
      nx = s.loff[bw];
      ny = s.loff[s.ul[q]];
    } else if (MODE == kSiOff) {
      const int zb = s.oz[q], qq = s.ol[q];
      nj = s.bs[s.colrow[qq]];
      nx = s.loff[zb < 0 ? ~zb : zb];
      if (zb < 0) nj = -nj;
      ny = s.loff[qq];
    } else {
      nj = -s.bs[s.colrow[q0 + q]];
      nx = ny = s.loff[q0 + q];
    }
  };
  const double* xall = MODE == kSiUpdate ? s.W : s.Z;
  fetch(t);
  wait_for_previous();
  for (; t < te; t += S) {
    const int n = (int)min((int64_t)S, te - t);
    const int mj = nj;
    const int64_t mx = nx, my = ny;
    const int widest = (int)__reduce_max_sync(0xffffffffu, (unsigned)abs(mj));
    for (int t0 = 0; t0 < widest; t0 += KC) {
      const int kc = min(KC, widest - t0), sx = th * kc, ss = sx + kc * tw;
      __syncwarp();
      for (int u = 0; u < n; ++u) {
        const int sj = __shfl_sync(0xffffffffu, mj, u), bj = abs(sj);
        const int64_t xo = __shfl_sync(0xffffffffu, mx, u), yo = __shfl_sync(0xffffffffu, my, u);
        const int kw = min(kc, bj - t0);
        if (kw <= 0) continue;
        const uint32_t d = sbase + 8u * (uint32_t)(u * ss);
        if (sj < 0) d64_stage(d, xall + xo + (int64_t)t0 * bi + r0, kw, th, bi, lane);
        else d64_stage(d, xall + xo + (int64_t)r0 * bj + t0, th, kw, bj, lane);
        if (kYRows) d64_stage(d + 8u * (uint32_t)sx, s.L + yo + (int64_t)c0 * bj + t0, tw, kw, bj, lane);
        else d64_stage(d + 8u * (uint32_t)sx, s.L + yo + (int64_t)t0 * bk + c0, kw, tw, bk, lane);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      if (t0 == 0) fetch(t + S);
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      __syncwarp();
      const int left = abs(mj) - t0;  // t extent left of this lane's term
      if (n * ne == used && __all_sync(0xffffffffu, lane >= n || left >= kc)) {
        // a full step of terms all as wide as the step: kSiChains slots' chains side by side
        const int live = (n * ne + 31) >> 5;
#pragma unroll
        for (int m0 = 0; m0 < kSiSlots; m0 += kSiChains) {
          if (m0 >= live) break;
          const double* xp[kSiChains];
          const double* yp[kSiChains];
          int xt[kSiChains];
#pragma unroll
          for (int v = 0; v < kSiChains; ++v) {
            const int o = off[min(m0 + v, kSiSlots - 1)], u = o >> 16, r = (o >> 8) & 255, c = o & 255;
            const bool tr = __shfl_sync(0xffffffffu, mj, u) < 0;
            xp[v] = base + u * ss + (tr ? r : r * kc);
            yp[v] = base + u * ss + sx + (kYRows ? c * kc : c);
            xt[v] = tr ? th : 1;
          }
#pragma unroll 2
          for (int tt = 0; tt < kc; ++tt) {
#pragma unroll
            for (int v = 0; v < kSiChains; ++v) {
              if (m0 + v < kSiSlots && m0 + v < live) acc[m0 + v] = fma(*xp[v], *yp[v], acc[m0 + v]);
              xp[v] += xt[v];
              yp[v] += kYRows ? 1 : tw;
            }
          }
        }
        continue;
      }
#pragma unroll
      for (int m = 0; m < kSiSlots; ++m) {
        if (32 * m >= n * ne) break;
        const int o = off[m], u = o >> 16, r = (o >> 8) & 255, c = o & 255;
        const int kl = max(0, min(kc, __shfl_sync(0xffffffffu, left, u)));  // 0 beyond the step
        const bool tr = __shfl_sync(0xffffffffu, mj, u) < 0;
        const int ku = (int)__reduce_max_sync(0xffffffffu, (unsigned)kl);
        const double* xp = base + u * ss + (tr ? r : r * kl);
        const double* yp = base + u * ss + sx + (kYRows ? c * kl : c);
        const int xt = tr ? th : 1;
        double v = acc[m];
#pragma unroll 2
        for (int tt = 0; tt < ku; ++tt, xp += xt, yp += kYRows ? 1 : tw)
          if (tt < kl) v = fma(*xp, *yp, v);
        acc[m] = v;
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int m = 0; m < kSiSlots; ++m)
    if (lane + 32 * m < used) base[lane + 32 * m] = acc[m];
  __syncwarp();
  for (int e = lane; e < ne; e += 32) {
    double v = used ? base[e] : 0.0;
    for (int u = ne; u < used; u += ne) v += base[u + e];
    base[e] = v;
  }
  __syncwarp();
}

// factor update W(i,k) = A(i,k) + sigma [i = k] - sum_j W(i,j) L(k,j)^T and inversion, off-diagonal
// blocks Z(i,k) = - sum_{j in struct(k)} Z(i,j) L(j,k).  parts = 0: a warp per item; else a CTA per
// item and part, its warps sharing the part; with parts > 1 the parts go to P.
template <int MODE>
__global__ void __launch_bounds__(kSiWarps * 32, 4) si_sum_kernel(SiDev s, const SiItem* __restrict__ items,
                                                                  int64_t nitems, int parts, int64_t E,
                                                                  const double* A, double sigma) {
  extern __shared__ __align__(16) double sh[];
  let_next_start();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t itn = parts ? (int64_t)(blockIdx.x / (unsigned)parts) : (int64_t)blockIdx.x * kSiWarps + w;
  if (itn >= nitems) return;  // (only whole warps of parts = 0)
  const int part = parts ? (int)(blockIdx.x % (unsigned)parts) : 0;
  const SiItem it = items[itn];
  const int i = s.colrow[it.blk], k = it.col;
  const int bi = s.bs[i], bk = s.bs[k];
  const int th = min(kTile, bi - it.r0), tw = min(kTile, bk - it.c0), ne = th * tw;
  const int64_t* ptr = MODE == kSiUpdate ? s.uptr : s.optr;
  const int64_t t0 = ptr[it.blk], nt = ptr[it.blk + 1] - t0;
  const int64_t ways = parts ? (int64_t)parts * kSiWarps : 1, me = parts ? (int64_t)part * kSiWarps + w : 0;
  si_sum<MODE>(s, t0 + nt * me / ways, t0 + nt * (me + 1) / ways, 0, bi, bk, it.r0, it.c0, th, tw,
               sh + (size_t)w * kSiBuf, lane);
  double* out = parts > 1 ? s.P + (int64_t)part * E + s.lpo[it.blk]
                          : (MODE == kSiUpdate ? s.W : s.Z) + s.loff[it.blk];
  const int64_t ao = MODE == kSiUpdate && part == 0 ? s.aoff[it.blk] : -1;
  if (parts) __syncthreads();
  for (int e = parts ? threadIdx.x : lane; e < ne; e += parts ? kSiWarps * 32 : 32) {
    double v = sh[(parts ? 0 : (size_t)w * kSiBuf) + e];
    if (parts)
      for (int u = 1; u < kSiWarps; ++u) v += sh[(size_t)u * kSiBuf + e];
    const int r = it.r0 + e / tw, c = it.c0 + e % tw;
    double b = 0.0;
    if (MODE == kSiUpdate && part == 0) {
      if (ao >= 0) b = A[ao + (int64_t)r * bk + c];
      if (i == k && r == c) b += sigma;
    }
    out[(int64_t)r * bk + c] = b - v;
  }
}

// Entry idx behind block q's first of the level's sums: W or Z itself, or the parts added in order.
__device__ __forceinline__ double si_assembled(const SiDev& s, const double* base, int64_t q, int64_t idx, int parts,
                                               int64_t E) {
  if (parts <= 1) return base[s.loff[q] + idx];
  const double* p = s.P + s.lpo[q] + idx;
  double v = p[0];
#pragma unroll 8
  for (int t = 1; t < parts; ++t) v += p[(int64_t)t * E];
  return v;
}

// pivot: D(k,k)^{-1} by Gauss-Jordan without pivoting, then L(i,k) = W(i,k) D(k,k)^{-1}.  A column's
// blocks lie one after the other with the same row pitch, so they are one tall matrix: CTA (x, y)
// serves supernode sn[x] and the rows y * rows .. of it below the diagonal block; y = 0 stores
// D^{-1}.  With parts > 1 the blocks are first assembled from the update's parts (and W(i,k)
// stored).  Each CTA inverts D for itself; an entry of D stays in one thread's register, a pivot
// step is one barrier and one division.
__global__ void __launch_bounds__(kSiThreads) si_pivot_kernel(SiDev s, const int32_t* __restrict__ sn, int parts,
                                                              int64_t E, int rows) {
  extern __shared__ __align__(16) double sh[];  // D^{-1}, then a chunk of W
  __shared__ double prow[2][kSiMaxB], pcol[2][kSiMaxB];
  const int k = sn[blockIdx.x];
  const int bk = s.bs[k], n2 = bk * bk, tid = threadIdx.x;
  const int64_t c0 = s.colptr[k], c1 = s.colptr[k + 1];
  const int64_t first = s.loff[c0] + n2, total = c1 > c0 + 1 ? s.loff[c1] - first : 0;  // entries below the diagonal
  const int64_t e0 = (int64_t)blockIdx.y * rows * bk, e1 = min(total, e0 + (int64_t)rows * bk);
  let_next_start();
  if (blockIdx.y > 0 && e0 >= total) return;
  wait_for_previous();
  double v[kSiMaxB * kSiMaxB / kSiThreads];
#pragma unroll
  for (int m = 0; m < kSiMaxB * kSiMaxB / kSiThreads; ++m) {
    if (m * kSiThreads >= n2) break;
    const int idx = tid + m * kSiThreads;
    if (idx < n2) v[m] = si_assembled(s, s.W, c0, idx, parts, E);
  }
  bool ok = true;
  for (int p = 0; p < bk; ++p) {
    double* pr = prow[p & 1];
    double* pc = pcol[p & 1];
#pragma unroll
    for (int m = 0; m < kSiMaxB * kSiMaxB / kSiThreads; ++m) {
      if (m * kSiThreads >= n2) break;
      const int idx = tid + m * kSiThreads;
      if (idx < n2) {
        const int r = idx / bk, c = idx - r * bk;
        if (r == p) pr[c] = v[m];
        if (c == p) pc[r] = v[m];
      }
    }
    __syncthreads();  // the buffers of step p are rewritten at p + 2, behind the barrier of p + 1
    const double piv = pr[p];
    if (!(piv > 0.0) || !isfinite(piv)) ok = false;
    const double inv = 1.0 / piv;
#pragma unroll
    for (int m = 0; m < kSiMaxB * kSiMaxB / kSiThreads; ++m) {
      if (m * kSiThreads >= n2) break;
      const int idx = tid + m * kSiThreads;
      if (idx < n2) {
        const int r = idx / bk, c = idx - r * bk;
        const double q = c == p ? inv : pr[c] * inv;
        v[m] = r == p ? q : (c == p ? 0.0 : v[m]) - pc[r] * q;
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kSiMaxB * kSiMaxB / kSiThreads; ++m) {
    if (m * kSiThreads >= n2) break;
    const int idx = tid + m * kSiThreads;
    if (idx < n2) {
      sh[idx] = v[m];
      if (blockIdx.y == 0) s.L[s.loff[c0] + idx] = v[m];
    }
  }
  if (blockIdx.y == 0 && !ok && tid == 0) {
    *(volatile unsigned int*)s.flag = 1u;
    __threadfence_system();
  }
  double* Wb = sh + n2;
  const int64_t step = kSiChunk / bk * bk;  // whole rows
  for (int64_t e = e0; e < e1; e += step) {
    const int len = (int)min(step, e1 - e);
    __syncthreads();
    for (int idx = tid; idx < len; idx += kSiThreads) {
      const double w = si_assembled(s, s.W, c0, n2 + e + idx, parts, E);
      Wb[idx] = w;
      if (parts > 1) s.W[first + e + idx] = w;
    }
    __syncthreads();
    for (int idx = tid; idx < len; idx += kSiThreads) {
      const int r = idx / bk, c = idx - r * bk;
      const double* wr = Wb + r * bk;
      double t = 0.0;
      for (int u = 0; u < bk; ++u) t = fma(wr[u], sh[u * bk + c], t);
      s.L[first + e + idx] = t;
    }
  }
}

// inversion, diagonal blocks: Z(k,k) = D^{-1} - sum_{j in struct(k)} Z(j,k)^T L(j,k).  A cluster of
// CTAs (one, or kSiCluster where a column of the level is long) serves a supernode: each CTA
// assembles its share of the Z(j,k) from the off-diagonal parts (parts > 1), its warps sum their
// terms, and the CTAs' sums are added in order through distributed shared memory.
__global__ void __launch_bounds__(kSiWarps * 32, 4) si_diag_kernel(SiDev s, const int32_t* __restrict__ sn, int parts,
                                                                   int64_t E) {
  extern __shared__ __align__(16) double sh[];
  __shared__ double csum[kTile * kTile];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = sn[blockIdx.x / (unsigned)ctas];
  const int bk = s.bs[k];
  const int64_t c0 = s.colptr[k] + 1, nt = s.colptr[k + 1] - c0;
  const int64_t t0 = nt * rank / ctas, t1 = nt * (rank + 1) / ctas;  // this CTA's terms
  let_next_start();
  wait_for_previous();
  if (parts > 1 && t1 > t0) {
    const int64_t z0 = s.loff[c0 + t0], len = s.loff[c0 + t1] - z0;
    for (int64_t idx = threadIdx.x; idx < len; idx += blockDim.x)
      s.Z[z0 + idx] = si_assembled(s, s.Z, c0 + t0, idx, parts, E);
    __syncthreads();
  }
  const double* Dinv = s.L + s.loff[c0 - 1];
  double* Zkk = s.Z + s.loff[c0 - 1];
  for (int r0 = 0; r0 < bk; r0 += kTile)
    for (int d0 = 0; d0 < bk; d0 += kTile) {
      const int th = min(kTile, bk - r0), tw = min(kTile, bk - d0), ne = th * tw;
      si_sum<kSiDiag>(s, t0 + (t1 - t0) * w / kSiWarps, t0 + (t1 - t0) * (w + 1) / kSiWarps, c0, bk, bk, r0, d0, th, tw,
                      sh + (size_t)w * kSiBuf, lane);
      __syncthreads();
      for (int e = threadIdx.x; e < ne; e += blockDim.x) {
        double v = sh[e];
        for (int u = 1; u < kSiWarps; ++u) v += sh[(size_t)u * kSiBuf + e];
        csum[e] = v;
      }
      cluster.sync();
      for (int e = rank * kSiWarps * 32 + threadIdx.x; e < ne; e += ctas * kSiWarps * 32) {
        double v = 0.0;
        for (int u = 0; u < ctas; ++u) v += cluster.map_shared_rank(csum, u)[e];
        const int at = (r0 + e / tw) * bk + d0 + e % tw;
        Zkk[at] = Dinv[at] - v;
      }
      cluster.sync();  // no CTA reuses its sums or leaves while another reads them
    }
}

// out = alpha P_S(Z) + beta out: one warp per block of S
__global__ void si_scatter_kernel(int64_t nblocks, const int32_t* __restrict__ sbsize,
                                  const int32_t* __restrict__ sbrow, const int32_t* __restrict__ scol,
                                  const int64_t* __restrict__ svoff, const int32_t* __restrict__ s2l,
                                  const int8_t* __restrict__ s2t, const int64_t* __restrict__ loff,
                                  const double* __restrict__ Z, double alpha, double beta, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nblocks;
       b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int br = sbsize[sbrow[b]], bc = sbsize[scol[b]];
    const int lb = s2l[b];
    if (lb < 0) continue;  // an empty block
    const bool tr = s2t[b] != 0;
    const double* zb = Z + loff[lb];
    double* o = out + svoff[b];
    for (int e = lane; e < br * bc; e += 32) {
      const int r = e / bc, c = e - r * bc;
      const double z = tr ? zb[(int64_t)c * br + r] : zb[e];
      o[e] = beta == 0.0 ? alpha * z : alpha * z + beta * o[e];
    }
  }
}

// ---- host: symbolic analysis ------------------------------------------------------------

struct Symbolic {
  int32_t m = 0;                         // non-empty clusters
  std::vector<int32_t> perm;             // position -> cluster (non-empty first)
  std::vector<int32_t> pos;              // cluster -> position (-1: empty cluster)
  std::vector<std::vector<int32_t>> st;  // struct(p): positions below p in column p, ascending
};

// Symmetric, sorted, in-range pattern check; returns S_ERR_PATTERN on a violation.
s_status check_symmetric(int32_t nc, const int64_t* rowptr, const int32_t* colidx) {
  for (int32_t r = 0; r < nc; ++r) {
    for (int64_t q = rowptr[r]; q < rowptr[r + 1]; ++q) {
      const int32_t c = colidx[q];
      if (c < 0 || c >= nc || (q > rowptr[r] && colidx[q - 1] >= c))
        return set_error(S_ERR_PATTERN, "selected inversion: pattern rows must be sorted and in range");
      const int32_t* b = colidx + rowptr[c];
      const int32_t* e = colidx + rowptr[c + 1];
      const int32_t* f = std::lower_bound(b, e, r);
      if (f == e || *f != r) return set_error(S_ERR_PATTERN, "selected inversion: the pattern is not symmetric");
    }
  }
  return S_OK;
}

// Minimum degree on the block graph (exact degrees, bitset rows), ties to the smaller id.
s_status symbolic(int32_t nc, const int64_t* rowptr, const int32_t* colidx, const int32_t* bsize, Symbolic* out) {
  s_status st = check_symmetric(nc, rowptr, colidx);
  if (st) return st;
  std::vector<int32_t> vid(nc, -1), cl;
  for (int32_t c = 0; c < nc; ++c)
    if (bsize[c] > 0) {
      vid[c] = (int32_t)cl.size();
      cl.push_back(c);
    }
  const int32_t m = (int32_t)cl.size();
  if (m > kSiMaxClusters) return set_error(S_ERR_ARG, "selected inversion: more than 32768 non-empty clusters");
  const int64_t W = (m + 63) / 64;
  std::vector<uint64_t> adj((size_t)m * W, 0ull), alive((size_t)W, 0ull);
  for (int32_t v = 0; v < m; ++v) alive[v >> 6] |= 1ull << (v & 63);
  for (int32_t v = 0; v < m; ++v) {
    const int32_t r = cl[v];
    for (int64_t q = rowptr[r]; q < rowptr[r + 1]; ++q) {
      const int32_t u = vid[colidx[q]];
      if (u >= 0 && u != v) adj[(size_t)v * W + (u >> 6)] |= 1ull << (u & 63);
    }
  }
  std::vector<int32_t> deg(m);
  for (int32_t v = 0; v < m; ++v) {
    int d = 0;
    for (int64_t w = 0; w < W; ++w) d += __builtin_popcountll(adj[(size_t)v * W + w]);
    deg[v] = d;
  }
  std::vector<uint8_t> done(m, 0);
  std::vector<int32_t> order;
  order.reserve(m);
  std::vector<std::vector<int32_t>> nbv(m);
  std::vector<int32_t> nb;
  for (int32_t step = 0; step < m; ++step) {
    int32_t v = -1;
    for (int32_t u = 0; u < m; ++u)
      if (!done[u] && (v < 0 || deg[u] < deg[v])) v = u;
    done[v] = 1;
    alive[v >> 6] &= ~(1ull << (v & 63));
    order.push_back(v);
    uint64_t* av = &adj[(size_t)v * W];
    nb.clear();
    for (int64_t w = 0; w < W; ++w) {
      uint64_t x = av[w] & alive[w];
      av[w] = x;
      while (x) {
        const int b = __builtin_ctzll(x);
        x &= x - 1;
        nb.push_back((int32_t)(w * 64 + b));
      }
    }
    nbv[v] = nb;
    for (int32_t u : nb) {
      uint64_t* au = &adj[(size_t)u * W];
      int d = 0;
      for (int64_t w = 0; w < W; ++w) {
        const uint64_t x = (au[w] | av[w]) & alive[w];
        au[w] = x;
        d += __builtin_popcountll(x);
      }
      au[u >> 6] &= ~(1ull << (u & 63));
      deg[u] = d - 1;  // the union held u itself (u is a neighbour of v)
    }
  }
  out->m = m;
  out->perm.assign(nc, 0);
  out->pos.assign(nc, -1);
  std::vector<int32_t> vpos(m);
  for (int32_t p = 0; p < m; ++p) {
    vpos[order[p]] = p;
    out->perm[p] = cl[order[p]];
    out->pos[cl[order[p]]] = p;
  }
  int32_t p = m;
  for (int32_t c = 0; c < nc; ++c)
    if (bsize[c] <= 0) out->perm[p++] = c;
  out->st.assign(m, {});
  for (int32_t q = 0; q < m; ++q) {
    const int32_t v = order[q];
    std::vector<int32_t>& s = out->st[q];
    s.reserve(nbv[v].size());
    for (int32_t u : nbv[v]) s.push_back(vpos[u]);
    std::sort(s.begin(), s.end());
  }
  return S_OK;
}

std::vector<int32_t> etree_levels(const Symbolic& sy, int32_t* height) {
  std::vector<int32_t> lvl(sy.m, 0);
  int32_t h = 0;
  for (int32_t p = 0; p < sy.m; ++p) {
    if (!sy.st[p].empty()) {
      const int32_t par = sy.st[p][0];
      lvl[par] = std::max(lvl[par], lvl[p] + 1);
    }
    h = std::max(h, lvl[p] + 1);
  }
  *height = sy.m ? h : 0;
  return lvl;
}

template <typename T>
s_status upload(T** dst, const std::vector<T>& v) {
  const cudaError_t e = cudaMalloc((void**)dst, sizeof(T) * std::max<size_t>(v.size(), 1));
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    *dst = nullptr;
    return set_error(S_ERR_NOMEM, "selected inversion: no device memory for the plan's lists");
  }
  SF_CUDA(e);
  if (!v.empty()) SF_CUDA(cudaMemcpy(*dst, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return S_OK;
}

// ---- host: elliptic functions for Eq. (ContInt) ------------------------------------------

// K(m) = pi / (2 AGM(1, sqrt(1 - m))), 0 <= m < 1.
double ellip_k(double m) {
  double a = 1.0, b = std::sqrt(1.0 - m);
  for (int it = 0; it < 64 && std::fabs(a - b) > 1e-16 * a; ++it) {
    const double an = 0.5 * (a + b);
    b = std::sqrt(a * b);
    a = an;
  }
  return M_PI / (a + b);
}

// sn, cn, dn(u|m) by the descending arithmetic-geometric mean (Abramowitz and Stegun 16.4):
// a_0 = 1, b_0 = sqrt(1-m), c_0 = sqrt(m); a_n, b_n the AGM steps, c_n = (a_{n-1} - b_{n-1})/2
// until c_N is negligible; phi_N = 2^N a_N u and phi_{n-1} = (phi_n + asin(c_n sin(phi_n)/a_n))/2;
// sn = sin phi_0, cn = cos phi_0, dn = cos phi_0 / cos(phi_1 - phi_0).
void ellip_j(double u, double m, double* sn, double* cn, double* dn) {
  if (m <= 0.0) {
    *sn = std::sin(u);
    *cn = std::cos(u);
    *dn = 1.0;
    return;
  }
  double a[40], c[40];
  a[0] = 1.0;
  double b = std::sqrt(1.0 - m);
  c[0] = std::sqrt(m);
  int n = 0;
  while (n < 38 && std::fabs(c[n]) > 1e-16) {
    a[n + 1] = 0.5 * (a[n] + b);
    c[n + 1] = 0.5 * (a[n] - b);
    b = std::sqrt(a[n] * b);
    ++n;
  }
  double phi = std::ldexp(a[n] * u, n);
  double prev = phi;
  for (int j = n; j >= 1; --j) {
    prev = phi;
    phi = 0.5 * (phi + std::asin(c[j] * std::sin(phi) / a[j]));
  }
  *sn = std::sin(phi);
  *cn = std::cos(phi);
  *dn = n >= 1 ? *cn / std::cos(prev - phi) : 1.0;
}

}  // namespace
}  // namespace sf

using namespace sf;

struct s_selinv_t {
  const s_pattern_t* S = nullptr;
  int32_t m = 0, height = 0, maxb = 0;
  int64_t nl = 0, nent = 0, nterms = 0;
  double flops_factor = 0.0, flops_invert = 0.0;
  // level lists (host offsets into the device arrays)
  std::vector<int64_t> upd_ptr, off_ptr, sn_ptr;
  std::vector<int32_t> lvl_rows, lvl_slices;  // rows of a pivot CTA, pivot CTAs per supernode
  std::vector<int64_t> lvl_longest;           // longest struct(k) of each level
  std::vector<int64_t> lvl_ent;               // entries of the blocks of each level's columns
  std::vector<int32_t> upd_parts, off_parts;  // 0: a warp per item, else CTAs per item
  // device
  int32_t* bs = nullptr;
  int64_t* colptr = nullptr;
  int32_t* colrow = nullptr;
  int64_t* loff = nullptr;
  int32_t* colcol = nullptr;
  int64_t* uptr = nullptr;
  int32_t* uw = nullptr;
  int32_t* ul = nullptr;
  int64_t* optr = nullptr;
  int32_t* oz = nullptr;
  int32_t* ol = nullptr;
  int64_t* aoff = nullptr;
  int64_t* lpo = nullptr;
  double* P = nullptr;
  SiItem* upd = nullptr;
  SiItem* off = nullptr;
  int32_t* sn = nullptr;
  int32_t* s2l = nullptr;
  int8_t* s2t = nullptr;
  double* W = nullptr;
  double* L = nullptr;
  double* Z = nullptr;
  unsigned int* flag = nullptr;
  unsigned int* flag_host = nullptr;
};

static void selinv_free(s_selinv_t* p) {
  cudaFree(p->bs);
  cudaFree(p->colptr);
  cudaFree(p->colrow);
  cudaFree(p->loff);
  cudaFree(p->colcol);
  cudaFree(p->uptr);
  cudaFree(p->uw);
  cudaFree(p->ul);
  cudaFree(p->optr);
  cudaFree(p->oz);
  cudaFree(p->ol);
  cudaFree(p->aoff);
  cudaFree(p->lpo);
  cudaFree(p->P);
  cudaFree(p->upd);
  cudaFree(p->off);
  cudaFree(p->sn);
  cudaFree(p->s2l);
  cudaFree(p->s2t);
  cudaFree(p->W);
  cudaFree(p->L);
  cudaFree(p->Z);
  if (p->flag_host) cudaFreeHost(p->flag_host);
}

static SiDev dev_of(const s_selinv_t* p) {
  SiDev s;
  s.bs = p->bs;
  s.colptr = p->colptr;
  s.colrow = p->colrow;
  s.loff = p->loff;
  s.colcol = p->colcol;
  s.uptr = p->uptr;
  s.uw = p->uw;
  s.ul = p->ul;
  s.optr = p->optr;
  s.oz = p->oz;
  s.ol = p->ol;
  s.aoff = p->aoff;
  s.lpo = p->lpo;
  s.W = p->W;
  s.L = p->L;
  s.Z = p->Z;
  s.P = p->P;
  s.flag = p->flag;
  return s;
}

static s_status selinv_build(s_selinv_t* p) {
  const s_pattern_t* S = p->S;
  const int32_t nc = (int32_t)S->bsize.size();
  Symbolic sy;
  s_status st = symbolic(nc, S->rowptr.data(), S->colidx.data(), S->bsize.data(), &sy);
  if (st) return st;
  const int32_t m = sy.m;
  p->m = m;
  std::vector<int32_t> lvl = etree_levels(sy, &p->height);
  std::vector<int32_t> bs(std::max(m, 1), 0);
  for (int32_t q = 0; q < m; ++q) {
    bs[q] = S->bsize[sy.perm[q]];
    if (bs[q] > kSiMaxB) return set_error(S_ERR_ARG, "selected inversion: blocks wider than 64");
    p->maxb = std::max(p->maxb, bs[q]);
  }
  // CSC of L
  std::vector<int64_t> colptr(m + 1, 0), loff;
  std::vector<int32_t> colrow;
  for (int32_t k = 0; k < m; ++k) colptr[k + 1] = colptr[k] + 1 + (int64_t)sy.st[k].size();
  const int64_t nl = colptr[m];
  if (nl >= INT32_MAX) return set_error(S_ERR_ARG, "selected inversion: factor has more than 2^31 blocks");
  colrow.reserve(nl);
  loff.reserve(nl + 1);
  int64_t e = 0;
  double ff = 0.0, fi = 0.0;
  for (int32_t k = 0; k < m; ++k) {
    colrow.push_back(k);
    loff.push_back(e);
    e += (int64_t)bs[k] * bs[k];
    double T = 0.0, T2 = 0.0;
    for (int32_t i : sy.st[k]) {
      colrow.push_back(i);
      loff.push_back(e);
      e += (int64_t)bs[i] * bs[k];
      T += bs[i];
      T2 += (double)bs[i] * bs[i];
    }
    const double b = bs[k];
    // update pairs (i >= i') of struct(k) and the pivot; inversion: struct(k) x struct(k)
    ff += b * (T * T + T2) + 2.0 * b * b * b + 2.0 * b * b * T;
    fi += 2.0 * b * T * T + 2.0 * b * b * T;
  }
  loff.push_back(e);
  p->nl = nl;
  p->nent = e;
  p->flops_factor = ff;
  p->flops_invert = fi;
  // CSR of L: row i holds its columns ascending (the diagonal last)
  std::vector<int64_t> rowptr(m + 1, 0);
  for (int64_t q = 0; q < nl; ++q) ++rowptr[colrow[q] + 1];
  for (int32_t i = 0; i < m; ++i) rowptr[i + 1] += rowptr[i];
  std::vector<int32_t> rowcol(nl), rowblk(nl);
  {
    std::vector<int64_t> fill(rowptr.begin(), rowptr.end() - 1);
    for (int32_t k = 0; k < m; ++k)
      for (int64_t q = colptr[k]; q < colptr[k + 1]; ++q) {
        const int32_t i = colrow[q];
        rowcol[fill[i]] = k;
        rowblk[fill[i]] = (int32_t)q;
        ++fill[i];
      }
  }
  // S blocks of each L block, and L blocks of each S block
  std::vector<int64_t> aoff(nl, -1);
  const int64_t snb = (int64_t)S->colidx.size();
  std::vector<int32_t> s2l(std::max<int64_t>(snb, 1), -1);
  std::vector<int8_t> s2t(std::max<int64_t>(snb, 1), 0);
  for (int32_t r = 0; r < nc; ++r) {
    for (int64_t b = S->rowptr[r]; b < S->rowptr[r + 1]; ++b) {
      const int32_t c = S->colidx[b];
      const int32_t pr = sy.pos[r], pc = sy.pos[c];
      if (pr < 0 || pc < 0) continue;
      const int32_t hi = std::max(pr, pc), lo = std::min(pr, pc);
      const int32_t* f = std::lower_bound(colrow.data() + colptr[lo], colrow.data() + colptr[lo + 1], hi);
      if (f == colrow.data() + colptr[lo + 1] || *f != hi)
        return set_error(S_ERR_PATTERN, "selected inversion: internal error, S not inside the factor");
      const int64_t q = f - colrow.data();
      s2l[b] = (int32_t)q;
      s2t[b] = pr < pc ? 1 : 0;
      if (pr >= pc) aoff[q] = S->voff[b];
    }
  }
  for (int32_t k = 0; k < m; ++k)
    if (aoff[colptr[k]] < 0) return set_error(S_ERR_PATTERN, "selected inversion: pattern lacks a diagonal block");
  // Term lists of both sweeps (fixed by the pattern of L), per CSC block q = (i,k):
  //   factor:    the j < k in both row i and row k of L, as CSC blocks W(i,j), L(k,j);
  //   inversion: (i > k) for every j in struct(k), the block holding Z(i,j) (~index when it is
  //              stored as Z(j,i)) and the block L(j,k).
  std::vector<int64_t> uptr(nl + 1, 0), optr(nl + 1, 0);
  std::vector<int32_t> uw, ul, oz, ol, colcol(nl);
  for (int32_t k = 0; k < m; ++k) {
    const int64_t rk0 = rowptr[k], rk1 = rowptr[k + 1] - 1;  // row k below its diagonal
    for (int64_t q = colptr[k]; q < colptr[k + 1]; ++q) {
      const int32_t i = colrow[q];
      colcol[q] = k;
      for (int64_t a = rowptr[i], ae = rowptr[i + 1], b = rk0; a < ae && b < rk1 && rowcol[a] < k;) {
        if (rowcol[a] < rowcol[b]) {
          ++a;
        } else if (rowcol[b] < rowcol[a]) {
          ++b;
        } else {
          uw.push_back(rowblk[a]);
          ul.push_back(rowblk[b]);
          ++a;
          ++b;
        }
      }
      uptr[q + 1] = (int64_t)uw.size();
      if (q > colptr[k]) {
        int64_t ra = rowptr[i], ca = colptr[i] + 1;
        const int64_t re = rowptr[i + 1], ce = colptr[i + 1];
        for (int64_t qq = colptr[k] + 1; qq < colptr[k + 1]; ++qq) {
          const int32_t j = colrow[qq];
          int32_t zb;
          if (j < i) {
            while (ra < re && rowcol[ra] < j) ++ra;
            if (ra == re || rowcol[ra] != j) return set_error(S_ERR_PATTERN, "selected inversion: internal error");
            zb = rowblk[ra];
          } else if (j == i) {
            zb = (int32_t)colptr[i];
          } else {
            while (ca < ce && colrow[ca] < j) ++ca;
            if (ca == ce || colrow[ca] != j) return set_error(S_ERR_PATTERN, "selected inversion: internal error");
            zb = ~(int32_t)ca;
          }
          oz.push_back(zb);
          ol.push_back((int32_t)qq);
        }
      }
      optr[q + 1] = (int64_t)oz.size();
    }
  }
  p->nterms = (int64_t)uw.size() + (int64_t)oz.size();
  // level lists, level-local entry offsets, and the split of each level's long sums
  const int32_t H = p->height;
  std::vector<std::vector<int32_t>> bylvl(H);
  for (int32_t k = 0; k < m; ++k) bylvl[lvl[k]].push_back(k);
  std::vector<SiItem> upd, off;
  std::vector<int32_t> sn;
  std::vector<int64_t> lpo(nl, 0);
  p->upd_ptr.assign(1, 0);
  p->off_ptr.assign(1, 0);
  p->sn_ptr.assign(1, 0);
  p->lvl_rows.assign(H, 1);
  p->lvl_slices.assign(H, 1);
  p->lvl_longest.assign(H, 0);
  p->lvl_ent.assign(H, 0);
  p->upd_parts.assign(H, 0);
  p->off_parts.assign(H, 0);
  const int64_t sms = sm_count();
  int64_t scratch = 0;
  for (int32_t l = 0; l < H; ++l) {
    int64_t longest = 0, ent = 0, maxu = 0, maxo = 0, rows = 0, maxrows = 0;
    const int64_t u0 = (int64_t)upd.size(), o0 = (int64_t)off.size();
    for (int32_t k : bylvl[l]) {
      sn.push_back(k);
      longest = std::max<int64_t>(longest, colptr[k + 1] - colptr[k] - 1);
      const int64_t below = (loff[colptr[k + 1]] - loff[colptr[k]]) / bs[k] - bs[k];
      rows += below;
      maxrows = std::max(maxrows, below);
      for (int64_t q = colptr[k]; q < colptr[k + 1]; ++q) {
        maxu = std::max<int64_t>(maxu, uptr[q + 1] - uptr[q]);
        maxo = std::max<int64_t>(maxo, optr[q + 1] - optr[q]);
        const int bi = bs[colrow[q]], bk = bs[k];
        lpo[q] = ent;
        ent += (int64_t)bi * bk;
        for (int r0 = 0; r0 < bi; r0 += kTile)
          for (int c0 = 0; c0 < bk; c0 += kTile) {
            upd.push_back(SiItem{(int32_t)q, k, (int16_t)r0, (int16_t)c0});
            if (q > colptr[k]) off.push_back(SiItem{(int32_t)q, k, (int16_t)r0, (int16_t)c0});
          }
      }
    }
    const int64_t nu = (int64_t)upd.size() - u0, no = (int64_t)off.size() - o0;
    // Ways of a level's sums.  A warp's terms take an SM sub-partition's FP64 pipe 1 us each (10 x 10
    // x 10), so a sum is spread until a warp holds kSiStepTerms of them or twice the resident
    // warps are at work; a warp per item only where the items alone fill the SMs.
    auto choose = [&](int64_t items, int64_t terms) -> int32_t {
      const int64_t slots = 2 * sms * 4;  // twice the resident CTAs
      if (items >= slots * kSiWarps || terms <= kSiStepTerms) return 0;
      int64_t q = std::min<int64_t>((slots + items - 1) / std::max<int64_t>(items, 1),
                                    (terms + kSiWarps * kSiStepTerms - 1) / (kSiWarps * kSiStepTerms));
      q = std::max<int64_t>(1, std::min<int64_t>(q, kSiMaxParts));
      while (q > 1 && q * ent > (int64_t)1 << 27) --q;  // scratch at most 1 GiB
      return (int32_t)q;
    };
    p->upd_parts[l] = choose(nu, maxu);
    p->off_parts[l] = choose(no, maxo);
    const int32_t parts = std::max(p->upd_parts[l], p->off_parts[l]);
    if (parts > 1) scratch = std::max<int64_t>(scratch, (int64_t)parts * ent);
    p->lvl_ent[l] = ent;
    p->lvl_longest[l] = longest;
    // pivot CTAs: 32 rows each while the level leaves SMs idle, up to 256
    p->lvl_rows[l] = (int32_t)std::min<int64_t>(256, std::max<int64_t>(32, (rows + sms * 4 - 1) / (sms * 4)));
    p->lvl_slices[l] = (int32_t)std::max<int64_t>(1, (maxrows + p->lvl_rows[l] - 1) / p->lvl_rows[l]);
    p->upd_ptr.push_back((int64_t)upd.size());
    p->off_ptr.push_back((int64_t)off.size());
    p->sn_ptr.push_back((int64_t)sn.size());
  }
  if ((st = upload(&p->bs, bs)) || (st = upload(&p->colptr, colptr)) || (st = upload(&p->colrow, colrow)) ||
      (st = upload(&p->loff, loff)) || (st = upload(&p->colcol, colcol)) || (st = upload(&p->uptr, uptr)) ||
      (st = upload(&p->uw, uw)) || (st = upload(&p->ul, ul)) || (st = upload(&p->optr, optr)) ||
      (st = upload(&p->oz, oz)) || (st = upload(&p->ol, ol)) || (st = upload(&p->aoff, aoff)) ||
      (st = upload(&p->lpo, lpo)) ||
      (st = upload(&p->upd, upd)) ||
      (st = upload(&p->off, off)) || (st = upload(&p->sn, sn)) || (st = upload(&p->s2l, s2l)) ||
      (st = upload(&p->s2t, s2t)))
    return st;
  const size_t vb = sizeof(double) * (size_t)std::max<int64_t>(e, 1);
  cudaError_t ce = cudaMalloc(&p->W, vb);
  if (ce == cudaSuccess) ce = cudaMalloc(&p->L, vb);
  if (ce == cudaSuccess) ce = cudaMalloc(&p->Z, vb);
  if (ce == cudaSuccess && scratch > 0) ce = cudaMalloc(&p->P, sizeof(double) * (size_t)scratch);
  if (ce == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return set_error(S_ERR_NOMEM, "selected inversion: no device memory for the factor");
  }
  SF_CUDA(ce);
  SF_CUDA(cudaHostAlloc((void**)&p->flag_host, sizeof(unsigned int), cudaHostAllocMapped));
  *(volatile unsigned int*)p->flag_host = 0u;
  SF_CUDA(cudaHostGetDevicePointer((void**)&p->flag, p->flag_host, 0));
  return S_OK;
}

extern "C" {

s_status s_selinv_order(int32_t n_clusters, const int64_t* rowptr, const int32_t* colidx, const int32_t* bsize,
                        int32_t* perm, int64_t* l_blocks, int32_t* levels) {
  if (n_clusters < 1 || !rowptr || !colidx || !bsize || !perm)
    return set_error(S_ERR_ARG, "s_selinv_order: null argument or no clusters");
  if (rowptr[0] != 0) return set_error(S_ERR_PATTERN, "s_selinv_order: rowptr[0] != 0");
  for (int32_t r = 0; r < n_clusters; ++r)
    if (rowptr[r + 1] < rowptr[r]) return set_error(S_ERR_PATTERN, "s_selinv_order: rowptr decreases");
  Symbolic sy;
  s_status st;
  try {
    st = symbolic(n_clusters, rowptr, colidx, bsize, &sy);
  } catch (const std::bad_alloc&) {
    st = set_error(S_ERR_NOMEM, "s_selinv_order: host memory exhausted");
  }
  if (st) return st;
  std::memcpy(perm, sy.perm.data(), sizeof(int32_t) * n_clusters);
  int64_t nl = sy.m;
  for (const auto& s : sy.st) nl += (int64_t)s.size();
  if (l_blocks) *l_blocks = nl;
  int32_t h = 0;
  etree_levels(sy, &h);
  if (levels) *levels = h;
  return S_OK;
}

s_status s_selinv_create(s_pattern S, s_selinv* out) {
  if (!S || !out) return set_error(S_ERR_ARG, "s_selinv_create: null argument");
  s_selinv_t* p = new s_selinv_t();
  p->S = S;
  s_status st;
  try {
    st = selinv_build(p);
  } catch (const std::bad_alloc&) {
    st = set_error(S_ERR_NOMEM, "selected inversion: host memory exhausted in the symbolic analysis");
  }
  if (st) {
    selinv_free(p);
    delete p;
    return st;
  }
  *out = p;
  return S_OK;
}

s_status s_selinv_destroy(s_selinv p) {
  if (!p) return S_OK;
  selinv_free(p);
  delete p;
  return S_OK;
}

s_status s_selinv_stats(s_selinv p, int64_t* l_blocks, int64_t* l_entries, int32_t* levels, double* flops_factor,
                        double* flops_invert) {
  if (!p) return set_error(S_ERR_ARG, "s_selinv_stats: null plan");
  if (l_blocks) *l_blocks = p->nl;
  if (l_entries) *l_entries = p->nent;
  if (levels) *levels = p->height;
  if (flops_factor) *flops_factor = p->flops_factor;
  if (flops_invert) *flops_invert = p->flops_invert;
  return S_OK;
}

// Dynamic shared memory of the sum kernels and of the pivot kernel (D^{-1} and a chunk of W).
constexpr size_t kSiSumBytes = sizeof(double) * kSiWarps * kSiBuf;
static size_t pivot_bytes(const s_selinv_t* p) { return sizeof(double) * ((size_t)p->maxb * p->maxb + kSiChunk); }

static s_status set_smem(const void* fn, size_t bytes) {
  if (bytes > 40 * 1024) SF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return S_OK;
}

s_status s_selinv_factor(s_selinv p, const double* A, double sigma, void* stream) {
  if (!p || (!A && p->S->d.nnz > 0)) return set_error(S_ERR_ARG, "s_selinv_factor: null argument");
  if (p->m == 0) return S_OK;
  cudaStream_t cs = (cudaStream_t)stream;
  const SiDev s = dev_of(p);
  s_status st;
  if ((st = set_smem((const void*)si_sum_kernel<kSiUpdate>, kSiSumBytes)) ||
      (st = set_smem((const void*)si_pivot_kernel, pivot_bytes(p))))
    return st;
  for (int32_t l = 0; l < p->height; ++l) {
    const int64_t n = p->upd_ptr[l + 1] - p->upd_ptr[l];
    const int parts = p->upd_parts[l];
    if (n > 0) {
      const int64_t grid = parts ? n * parts : (n + kSiWarps - 1) / kSiWarps;
      SF_CUDA(launch_overlapped(si_sum_kernel<kSiUpdate>, dim3((unsigned)grid), kSiWarps * 32, kSiSumBytes, 0, cs, s,
                        p->upd + p->upd_ptr[l], n, parts, p->lvl_ent[l], A, sigma));
    }
    const int64_t ns = p->sn_ptr[l + 1] - p->sn_ptr[l];
    if (ns > 0) {
      dim3 g((unsigned)ns, (unsigned)p->lvl_slices[l]);
      SF_CUDA(launch_overlapped(si_pivot_kernel, g, kSiThreads, pivot_bytes(p), 0, cs, s, p->sn + p->sn_ptr[l], parts,
                        p->lvl_ent[l], p->lvl_rows[l]));
    }
  }
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

s_status s_selinv_invert(s_selinv p, double alpha, double beta, double* out, void* stream) {
  if (!p || (!out && p->S->d.nnz > 0)) return set_error(S_ERR_ARG, "s_selinv_invert: null argument");
  cudaStream_t cs = (cudaStream_t)stream;
  if (p->m > 0) {
    const SiDev s = dev_of(p);
    s_status st;
    if ((st = set_smem((const void*)si_sum_kernel<kSiOff>, kSiSumBytes)) ||
        (st = set_smem((const void*)si_diag_kernel, kSiSumBytes)))
      return st;
    for (int32_t l = p->height - 1; l >= 0; --l) {
      const int64_t n = p->off_ptr[l + 1] - p->off_ptr[l];
      const int parts = p->off_parts[l];
      if (n > 0) {
        const int64_t grid = parts ? n * parts : (n + kSiWarps - 1) / kSiWarps;
        SF_CUDA(launch_overlapped(si_sum_kernel<kSiOff>, dim3((unsigned)grid), kSiWarps * 32, kSiSumBytes, 0, cs, s,
                          p->off + p->off_ptr[l], n, parts, p->lvl_ent[l], (const double*)nullptr, 0.0));
      }
      const int64_t ns = p->sn_ptr[l + 1] - p->sn_ptr[l];
      if (ns > 0) {
        // as many CTAs to a cluster as hold kSiStepTerms terms a warp and fit the SMs together
        unsigned ctas = 1;
        while (ctas < kSiCluster && p->lvl_longest[l] > (int64_t)ctas * kSiWarps * kSiStepTerms &&
               2 * ctas * ns <= (int64_t)sm_count() * 4)
          ctas *= 2;
        SF_CUDA(launch_overlapped(si_diag_kernel, dim3((unsigned)ns * ctas), kSiWarps * 32, kSiSumBytes, ctas, cs, s,
                          p->sn + p->sn_ptr[l], parts, p->lvl_ent[l]));
      }
    }
  }
  const DevPattern& d = p->S->d;
  if (d.nblocks > 0) {
    const int64_t grid = std::min<int64_t>((d.nblocks * 32 + 255) / 256, (int64_t)sm_count() * 8);
    si_scatter_kernel<<<(unsigned)std::max<int64_t>(grid, 1), 256, 0, cs>>>(
        d.nblocks, d.bsize, d.brow, d.colidx, d.voff, p->s2l, p->s2t, p->loff, p->Z, alpha, beta, out);
  }
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

s_status s_selinv_status(s_selinv p, void* stream) {
  if (!p) return set_error(S_ERR_ARG, "s_selinv_status: null plan");
  SF_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
  volatile unsigned int* w = p->flag_host;
  if (w && *w) {
    *w = 0u;
    return set_error(S_ERR_NOT_SPD, "selected inversion: a pivot block was not positive definite");
  }
  return S_OK;
}

s_status s_contour_nodes(double c_lo, double c_hi, int32_t n, double* shifts, double* weights) {
  if (!(c_lo > 0.0) || !(c_hi >= c_lo) || !std::isfinite(c_hi) || n < 1 || !shifts || !weights)
    return set_error(S_ERR_ARG, "s_contour_nodes: need 0 < c_lo <= c_hi and n >= 1");
  const double m = 1.0 - c_lo / c_hi;
  const double K = ellip_k(m);
  const double sc = std::sqrt(c_lo);
  for (int32_t k = 0; k < n; ++k) {
    const double t = K * (k + 0.5) / n;
    double sn, cn, dn;
    ellip_j(t, m, &sn, &cn, &dn);
    const double w = sc * sn / cn;
    shifts[k] = w * w;
    weights[k] = 2.0 * K * sc / (M_PI * n) * dn / (cn * cn);
  }
  return S_OK;
}

s_status s_selinv_invsqrt(s_selinv p, const double* A, double c_lo, double c_hi, int32_t n, double* out,
                          void* stream) {
  if (!p || n < 1 || n > 1024) return set_error(S_ERR_ARG, "s_selinv_invsqrt: null plan or n outside 1..1024");
  std::vector<double> w2(n), wt(n);
  s_status st = s_contour_nodes(c_lo, c_hi, n, w2.data(), wt.data());
  if (st) return st;
  for (int32_t k = 0; k < n; ++k) {
    if ((st = s_selinv_factor(p, A, w2[k], stream))) return st;
    if ((st = s_selinv_invert(p, wt[k], k ? 1.0 : 0.0, out, stream))) return st;
  }
  return s_selinv_status(p, stream);
}

}  // extern "C"
