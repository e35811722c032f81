// Streaming kernels on S-format value buffers: C = alpha A + beta B + gamma I (addition on
// a common pattern, Sec. 4.1), block-sparse matrix times vectors, and the power iteration and
// reductions of the norm estimate and the drivers.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace sf {

template <typename T>
__global__ void axpby_kernel(int64_t n, T alpha, const T* __restrict__ A, T beta, const T* __restrict__ B,
                             T* __restrict__ C) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
    T v = alpha * A[i];
    if (B) v = fma(beta, B[i], v);
    C[i] = v;
  }
}

template <typename T>
__global__ void add_diag_kernel(int32_t nc, const int32_t* diag, const int32_t* bsize, const int64_t* voff, T gamma,
                                T* C) {
  const int32_t nu = blockIdx.x;
  if (nu >= nc) return;
  const int k = diag[nu];
  if (k < 0) return;
  const int n = bsize[nu];
  for (int r = threadIdx.x; r < n; r += blockDim.x) C[voff[k] + (int64_t)r * n + r] += gamma;
}

static int grid_for(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8));
}

s_status run_add(const s_pattern_t* p, s_prec prec, double alpha, const void* A, double beta, const void* B,
                 double gamma, void* C, cudaStream_t st) {
  const int64_t n = p->d.nnz;
  if (gamma != 0.0 && !p->has_all_diag) return set_error(S_ERR_PATTERN, "s_add: gamma*I needs every diagonal block");
  if (prec == S_FP64) {
    if (n) axpby_kernel<double><<<grid_for(n), 256, 0, st>>>(n, alpha, (const double*)A, beta, (const double*)B, (double*)C);
    if (gamma != 0.0)
      add_diag_kernel<double><<<p->d.nc, 64, 0, st>>>(p->d.nc, p->d.diag, p->d.bsize, p->d.voff, gamma, (double*)C);
  } else if (prec == S_FP32) {
    if (n)
      axpby_kernel<float><<<grid_for(n), 256, 0, st>>>(n, (float)alpha, (const float*)A, (float)beta, (const float*)B,
                                                       (float*)C);
    if (gamma != 0.0)
      add_diag_kernel<float><<<p->d.nc, 64, 0, st>>>(p->d.nc, p->d.diag, p->d.bsize, p->d.voff, (float)gamma, (float*)C);
  } else {
    return set_error(S_ERR_ARG, "s_add: prec must be S_FP64 or S_FP32");
  }
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

// Y = A X for nvec vectors: the block rows by falling length, clusters of 8 CTAs of 4 warps.  A long
// row (more than kLongRow blocks) takes a whole cluster, the others one CTA each; the row's
// warps take several of its blocks at a time and deal the (block, row) pairs to their lanes, up
// to kSpPairs a lane with KV vectors each: a lane reads its row of the block once and multiplies
// it with the vectors.  The pairs' sums, then the warps', then the CTAs' (through distributed
// shared memory), are added in a fixed order.  What bounds it: for several vectors the FP64 pipe
// (2 nnz nvec operations, nearly all lanes at work), for one vector the loads; the root's row,
// which meets every cluster, is why long rows are shared (from 256 blocks on: from 64 or 128 the
// clusters' fixed cost took 1.2 to 1.8 times as long; but from 32 on in a matrix of at most two rows
// per SM, where a row's one CTA is a long chain on an idle GPU: space, 20-wide, N = 1000, one vector
// 47 -> 18 us, 16 vectors 328 -> 131 us, the same from 16 on).  Measured, N = 60000 in the plane, 10
// vectors (in brackets one thread per row and vector, A read once per vector): 1.30 ms (21.4), one
// vector 0.26 ms (2.14); five pairs a lane took 1.60 ms, staging blocks and vectors in shared
// memory as the double product does 1.33 ms and for one vector 0.47 ms.
constexpr int kSpWarps = 4;
constexpr int kSpCtas = 8;     // CTAs of a cluster
constexpr int kSpPairs = 3;    // (block, row) pairs of a lane
constexpr int kSpRows = 32;    // rows at a time
constexpr int kSpVec = 10;     // vectors at a time

template <int KV>
__global__ void __cluster_dims__(kSpCtas, 1, 1) __launch_bounds__(kSpWarps * 32, KV > 4 ? 4 : 6)
    spmm_kernel(int32_t nc, int32_t nlong, const int32_t* __restrict__ order, const int32_t* __restrict__ bsize,
                const int64_t* __restrict__ boff, const int64_t* __restrict__ rowptr,
                const int32_t* __restrict__ colidx, const int64_t* __restrict__ voff, const double* __restrict__ A,
                const double* __restrict__ X, int64_t n, int kv, double* __restrict__ Y) {
  __shared__ double psum[kSpWarps][32 * kSpPairs];
  __shared__ double wsum[kSpWarps][kSpRows * KV];
  __shared__ double csum[kSpRows * KV];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), cid = (int)(blockIdx.x / kSpCtas);
  const bool shared_row = cid < nlong;
  const int64_t at = shared_row ? cid : nlong + (int64_t)(cid - nlong) * kSpCtas + rank;
  if (at >= nc) return;  // (never in a cluster that shares a row)
  const int nu = order[at];
  const int ni = bsize[nu];
  const int64_t k0 = rowptr[nu], k1 = rowptr[nu + 1], row0 = boff[nu];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = shared_row ? kSpCtas * kSpWarps : kSpWarps, me = shared_row ? rank * kSpWarps + w : w;
  for (int r0 = 0; r0 < ni; r0 += kSpRows) {
    const int th = min(kSpRows, ni - r0);
    // blocks to a step: what the lanes hold, at most the warp's share of the row
    const int S = (int)max((int64_t)1, min((int64_t)(32 * kSpPairs / th), (k1 - k0 + nw - 1) / nw));
    double acc[kSpPairs][KV];
    int sp[kSpPairs], rp[kSpPairs];  // the lane's pairs: block of the step, row
#pragma unroll
    for (int m = 0; m < kSpPairs; ++m) {
      const int i = lane + 32 * m;
      sp[m] = i / th;
      rp[m] = i - sp[m] * th;
#pragma unroll
      for (int v = 0; v < KV; ++v) acc[m][v] = 0.0;
    }
    for (int64_t kb = k0 + (int64_t)me * S; kb < k1; kb += (int64_t)nw * S) {
      const int cnt = (int)min((int64_t)S, k1 - kb);
#pragma unroll
      for (int m = 0; m < kSpPairs; ++m) {
        if (sp[m] >= cnt) continue;
        const int64_t k = kb + sp[m];
        const int j = __ldg(colidx + k), nl = __ldg(bsize + j);
        const double* ap = A + __ldg(voff + k) + (int64_t)(r0 + rp[m]) * nl;
        const double* xp = X + __ldg(boff + j);
#pragma unroll 2
        for (int t = 0; t < nl; ++t) {
          const double e = ap[t];
#pragma unroll
          for (int v = 0; v < KV; ++v)
            if (v < kv) acc[m][v] = fma(e, __ldg(xp + (int64_t)v * n + t), acc[m][v]);
        }
      }
    }
    // the pairs of a row, then the warps, then the CTAs, each in order
#pragma unroll
    for (int v = 0; v < KV; ++v) {
      if (v >= kv) break;
#pragma unroll
      for (int m = 0; m < kSpPairs; ++m) psum[w][lane + 32 * m] = acc[m][v];
      __syncwarp();
      if (lane < th) {
        double q = 0.0;
        for (int s = 0; s < S; ++s) q += psum[w][s * th + lane];
        wsum[w][v * th + lane] = q;
      }
      __syncwarp();
    }
    __syncthreads();
    for (int e = threadIdx.x; e < th * kv; e += blockDim.x) {
      double q = wsum[0][e];
      for (int u = 1; u < kSpWarps; ++u) q += wsum[u][e];
      const int v = e / th;
      if (shared_row) csum[e] = q;
      else Y[(int64_t)v * n + row0 + r0 + (e - v * th)] = q;
    }
    if (shared_row) {
      cluster.sync();
      for (int e = rank * kSpWarps * 32 + threadIdx.x; e < th * kv; e += kSpCtas * kSpWarps * 32) {
        double q = 0.0;
        for (int u = 0; u < kSpCtas; ++u) q += cluster.map_shared_rank(csum, u)[e];
        const int v = e / th;
        Y[(int64_t)v * n + row0 + r0 + (e - v * th)] = q;
      }
      cluster.sync();  // no CTA reuses its sums or leaves while another reads them
    } else {
      __syncthreads();
    }
  }
}

s_status run_spmm_f64(const s_pattern_t* p, const double* A, const double* X, int nvec, double* Y, cudaStream_t st) {
  const DevPattern& d = p->d;
  if (nvec <= 0 || d.n == 0) return S_OK;
  const int64_t clusters = d.nlong + ((int64_t)d.nc - d.nlong + kSpCtas - 1) / kSpCtas;
  const int chunks = (nvec + kSpVec - 1) / kSpVec, most = (nvec + chunks - 1) / chunks;
  for (int v0 = 0; v0 < nvec; v0 += most) {
    const int kv = std::min(most, nvec - v0);
    auto kern = kv == 1   ? spmm_kernel<1>
                : kv == 2 ? spmm_kernel<2>
                : kv <= 4 ? spmm_kernel<4>
                : kv <= 6 ? spmm_kernel<6>
                : kv <= 8 ? spmm_kernel<8>
                          : spmm_kernel<kSpVec>;
    kern<<<(unsigned)(clusters * kSpCtas), kSpWarps * 32, 0, st>>>(d.nc, d.nlong, d.roworder, d.bsize, d.boff, d.rowptr,
                                                                   d.colidx, d.voff, A, X + (int64_t)v0 * d.n, d.n, kv,
                                                                   Y + (int64_t)v0 * d.n);
  }
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

// Sum of a thread's s over the CTA (256 threads) in a fixed order, in thread 0.
__device__ __forceinline__ double cta_sum(double s, double* red) {
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double v = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < (int)blockDim.x >> 5; ++q) v += red[q];
  __syncthreads();
  return v;
}

// part[cta] = sum of a b, part[kRedCtas + cta] = sum of b b over the CTA's share.  HBM-bound;
// one CTA for the whole vector takes 2 ms for 10^7 entries.
__global__ void __launch_bounds__(256) dot2_kernel(int64_t n, const double* __restrict__ a, const double* __restrict__ b,
                                                   double* __restrict__ part) {
  __shared__ double red[8];
  double s = 0.0, q = 0.0;
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (int64_t)kRedCtas * 256) {
    const double v = b[i];
    s = fma(a[i], v, s);
    q = fma(v, v, q);
  }
  s = cta_sum(s, red);
  q = cta_sum(q, red);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s;
    part[kRedCtas + blockIdx.x] = q;
  }
}

__global__ void __launch_bounds__(256) sum_kernel(int64_t n, const double* __restrict__ a, double* __restrict__ part) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (int64_t)kRedCtas * 256) s += a[i];
  s = cta_sum(s, red);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

s_status run_dot2(int64_t n, const double* a, const double* b, double* part, cudaStream_t st) {
  dot2_kernel<<<kRedCtas, 256, 0, st>>>(n, a, b, part);
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

s_status run_sum(int64_t n, const double* a, double* part, cudaStream_t st) {
  sum_kernel<<<kRedCtas, 256, 0, st>>>(n, a, part);
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

__global__ void power_start_kernel(int64_t n, double v, double* x, double* sc) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] = v;
  if (blockIdx.x == 0 && threadIdx.x < 2) sc[threadIdx.x] = 0.0;
}

// sc[0] = x.y, sc[1] = y.y from the partial sums (every CTA adds them, CTA 0 stores them), then
// x = y / sqrt(y.y); x unchanged when y = 0
__global__ void __launch_bounds__(256) power_scale_kernel(int64_t n, const double* __restrict__ y,
                                                          const double* __restrict__ part, double* __restrict__ x,
                                                          double* __restrict__ sc) {
  __shared__ double red[8], yy;
  const double q = cta_sum(part[kRedCtas + threadIdx.x], red);
  if (threadIdx.x == 0) yy = q;
  if (blockIdx.x == 0) {
    const double r = cta_sum(part[threadIdx.x], red);
    if (threadIdx.x == 0) {
      sc[0] = r;
      sc[1] = q;
    }
  }
  __syncthreads();
  const double s = yy;
  if (s <= 0.0) return;
  const double inv = 1.0 / sqrt(s);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = y[i] * inv;
}
static_assert(kRedCtas == 256, "power_scale_kernel adds one partial sum per thread");

s_status run_power(const s_pattern_t* p, const double* A, int iters, double* x, double* y, double* sc, cudaStream_t st) {
  const int64_t n = p->d.n;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 4));
  power_start_kernel<<<grid, 256, 0, st>>>(n, 1.0 / std::sqrt((double)n), x, sc);
  for (int it = 0; it < iters; ++it) {
    s_status s = run_spmm_f64(p, A, x, 1, y, st);
    if (s || (s = run_dot2(n, x, y, sc + 2, st))) return s;
    power_scale_kernel<<<grid, 256, 0, st>>>(n, y, sc + 2, x, sc);
  }
  SF_CUDA(cudaGetLastError());
  return S_OK;
}

}  // namespace sf

using namespace sf;

extern "C" s_status s_spmm(s_pattern p, const double* A, const double* X, int nvec, double* Y, void* stream) {
  if (!p || !A || !X || !Y || nvec < 0) return set_error(S_ERR_ARG, "s_spmm: bad argument");
  if (X == Y) return set_error(S_ERR_ARG, "s_spmm: Y aliases X");
  return run_spmm_f64(p, A, X, nvec, Y, (cudaStream_t)stream);
}

extern "C" s_status s_add(s_pattern p, s_prec prec, double alpha, const void* A, double beta, const void* B,
                          double gamma, void* C, void* stream) {
  if (!p || !A || !C || (beta != 0.0 && !B)) return set_error(S_ERR_ARG, "s_add: NULL argument");
  return run_add(p, prec, alpha, A, beta, beta != 0.0 ? B : nullptr, gamma, C, (cudaStream_t)stream);
}
