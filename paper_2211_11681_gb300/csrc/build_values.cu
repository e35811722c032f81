// Input preparation on the device: K^eta = P_S(T K T^T) (Thm. (S-compression)) for a
// Matern kernel (Sec. 2), exactly (all N^2 kernel evaluations) in float arithmetic, with
// the a-posteriori threshold of Sec. 5.
//
// Columns are processed in chunks: a chunk is a maximal cluster g with at most kChunk
// points.  For a chunk, U = K(all points, points of g) (N x |g|, tree order) is evaluated
// and transformed in place by the two-scale matrices Q of Eq. (QR): first along the
// columns inside g's subtree, then along all rows, level by level (the "slots" of a
// cluster are the rows/columns its transform reads and writes).  Afterwards U holds
// T K T_g^T: every block (a, b) of the pattern with b in g's subtree and a <= b is copied
// to an upper-triangle staging buffer together with its largest |entry|.  g's scaling
// columns are kept for the clusters above the chunks, which are then transformed and
// extracted the same way from the sons' scaling columns.  Finally the kept pattern is
// decided per unordered block pair and the values are assembled in double.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "build_internal.h"
#include "common.cuh"

namespace sf {

constexpr int kChunk = 1024;   // columns per chunk
constexpr int kRowTile = 16;   // rows per CTA of the evaluation kernel
constexpr int kColTile = 128;  // columns per CTA of the row transform
constexpr int kMaxIn = 64;     // largest n_in handled by the transform kernels

struct Geo {
  const float* x;          // N x 3 points in tree order
  const float* Q;          // all Q matrices, float, row-major nin x nin at qoff[c]
  const int64_t* qoff;
  const int32_t* slots;    // tree-order positions, slot_off[c] .. + nin(c)
  const int64_t* slot_off;
  const int32_t* nin;
  const int32_t* ns;
};

__device__ __forceinline__ float matern(float r, int p, float inv_ell, float scale) {
  // half-integer closed form, Sec. 2: nu = p + 1/2; p >= 3 encodes d/dell of nu = (p-3) + 1/2
  if (p >= 3) {
    // kappa = f(t), t = sqrt(2 nu) r / ell, dkappa/dell = -f'(t) t / ell
    const int q = p - 3;
    const float a = q == 0 ? 1.0f : (q == 1 ? 1.7320508075688772f : 2.23606797749979f);
    const float t = a * r * inv_ell;
    const float e = __expf(-t);
    float g;  // -f'(t) * t
    if (q == 0) g = t * e;
    else if (q == 1) g = t * t * e;
    else g = t * t * (1.0f + t) * (1.0f / 3.0f) * e;
    return scale * g * inv_ell;
  }
  if (p == 0) return scale * __expf(-r * inv_ell);
  if (p == 1) {
    const float t = 1.7320508075688772f * r * inv_ell;
    return scale * (1.0f + t) * __expf(-t);
  }
  const float t = 2.23606797749979f * r * inv_ell;
  return scale * (1.0f + t + t * t * (1.0f / 3.0f)) * __expf(-t);
}

// K(rows i0.., chunk columns) into shared memory, then the column transforms of every
// cluster of the chunk's subtree (bottom-up), then the tile to U (row-major N x w).
//
// The tile is held [column][kRowTile rows]: a half-warp applies a cluster's transform to 8 of the
// 16 rows, a lane to two of its columns at a time, so an input column's 8 values are two 16-byte
// broadcast loads and a step over one input is 16 multiply-adds a lane (with the tile
// [row][column] it was one multiply-add per two loads, one row at a time).  What bounds it: the
// 128 bytes a clock that shared memory delivers to registers.  Every sum runs over the inputs in
// ascending order.  Measured, N = 40000 on the sphere (nin 16 and 20), all chunks: 26.4 ms (one row
// at a time 79.6).
__global__ void __launch_bounds__(256) eval_colfwt_kernel(Geo g, int64_t n, int64_t q0, int w,
                                                          const int32_t* __restrict__ sub,
                                                          const int32_t* __restrict__ sub_lvl_off, int nlev, int p,
                                                          float inv_ell, float scale, int maxm, float* __restrict__ U) {
  extern __shared__ __align__(16) float tile[];  // w x kRowTile, then per warp Q (maxm x even pitch) and slots (maxm)
  const int64_t i0 = (int64_t)blockIdx.x * kRowTile;
  const int rows = (int)min((int64_t)kRowTile, n - i0);
  for (int e = threadIdx.x; e < kRowTile * w; e += blockDim.x) {
    const int r = e % kRowTile, j = e / kRowTile;
    float v = 0.0f;
    if (r < rows) {
      const float* xi = g.x + (i0 + r) * 3;
      const float* xj = g.x + (q0 + j) * 3;
      const float dx = xi[0] - xj[0], dy = xi[1] - xj[1], dz = xi[2] - xj[2];
      v = matern(sqrtf(dx * dx + dy * dy + dz * dz), p, inv_ell, scale);
    }
    tile[e] = v;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  // per warp: the cluster's Q (rows at an even pitch) and slots, staged once and applied to every row
  const int mp = (maxm + 1) & ~1;
  float* qs = tile + kRowTile * w + warp * (maxm * mp + mp);
  int* ss = reinterpret_cast<int*>(qs + maxm * mp);
  const int half = lane >> 4, hl = lane & 15;
  for (int L = 0; L < nlev; ++L) {  // sub is ordered deepest level first
    const int c0 = sub_lvl_off[L], c1 = sub_lvl_off[L + 1];
    for (int ci = c0 + warp; ci < c1; ci += nwarp) {
      const int c = sub[ci];
      const int m = g.nin[c];
      const int32_t* sl = g.slots + g.slot_off[c];
      const float* Q = g.Q + g.qoff[c];
      const float rm = 1.0f / (float)m;
      for (int e = lane; e < m * m; e += 32) {
        const int ii = __float2int_rz(((float)e + 0.5f) * rm);
        qs[ii * mp + (e - ii * m)] = Q[e];
      }
      for (int e = lane; e < m; e += 32) ss[e] = (sl[e] - (int)q0) * kRowTile;
      __syncwarp();
      // outputs j, j + 1 of this lane, at most two rounds of 16 lanes (m <= 64): kept until every
      // input has been read
      float o[2][2][8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int j = 2 * (hl + 16 * u);
        if (2 * 16 * u >= m) break;
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int r = 0; r < 8; ++r) o[u][v][r] = 0.0f;
        if (j < m) {
          const float* qj = qs + j;
          for (int ii = 0; ii < m; ++ii) {
            const float4* in = reinterpret_cast<const float4*>(tile + ss[ii] + 8 * half);
            const float4 a = in[0], b = in[1];
            const float2 q = *reinterpret_cast<const float2*>(qj + ii * mp);
            const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              o[u][0][r] = fmaf(x[r], q.x, o[u][0][r]);
              o[u][1][r] = fmaf(x[r], q.y, o[u][1][r]);
            }
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int j = 2 * (hl + 16 * u) + v;
          if (j < m) {
            float4* out = reinterpret_cast<float4*>(tile + ss[j] + 8 * half);
            out[0] = make_float4(o[u][v][0], o[u][v][1], o[u][v][2], o[u][v][3]);
            out[1] = make_float4(o[u][v][4], o[u][v][5], o[u][v][6], o[u][v][7]);
          }
        }
      __syncwarp();
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < (kRowTile / 4) * w; e += blockDim.x) {
    const int j = e % w, r = 4 * (e / w);
    const float4 v = *reinterpret_cast<const float4*>(tile + j * kRowTile + r);
    float* u = U + (i0 + r) * w + j;
    if (r < rows) u[0] = v.x;
    if (r + 1 < rows) u[w] = v.y;
    if (r + 2 < rows) u[2 * (int64_t)w] = v.z;
    if (r + 3 < rows) u[3 * (int64_t)w] = v.w;
  }
}

// In-place row transform of one level: rows slots(c) of U (ld w) <- Q_c^T rows.  A warp owns 32 VEC
// columns of a cluster and holds all their inputs in registers (MAXM of them), so the outputs go
// straight back; Q is staged once per CTA, which takes all columns of its cluster where they fit 8
// warps, and read four outputs at a time.  HBM / L2-bound: one read
// and one write of the rows it transforms.  Every sum runs over the inputs in
// ascending order.  Measured, N = 40000 on the sphere, all chunks and levels: 26.3 ms (through
// shared memory, 128 columns a CTA: 36.8).
template <int MAXM, int VEC>
__global__ void __launch_bounds__(256) rowfwt_reg_kernel(Geo g, const int32_t* __restrict__ lvl, int w,
                                                         float* __restrict__ U) {
  __shared__ __align__(16) float Qs[MAXM * MAXM];
  __shared__ int ss[MAXM];
  const int c = lvl[blockIdx.x];
  const int m = g.nin[c];
  const int32_t* sl = g.slots + g.slot_off[c];
  const float* Q = g.Q + g.qoff[c];
  for (int e = threadIdx.x; e < m * MAXM; e += blockDim.x) {
    const int ii = e / MAXM, jj = e - ii * MAXM;
    Qs[e] = jj < m ? Q[ii * m + jj] : 0.0f;
  }
  for (int e = threadIdx.x; e < m; e += blockDim.x) ss[e] = sl[e];
  __syncthreads();
  const int j0 = ((int)(blockIdx.y * blockDim.x + threadIdx.x) >> 5) * 32 * VEC + (int)(threadIdx.x & 31);
  if (j0 - (int)(threadIdx.x & 31) >= w) return;
  float in[MAXM][VEC];
#pragma unroll
  for (int ii = 0; ii < MAXM; ++ii) {
    if (ii < m) {
      const float* u = U + (int64_t)ss[ii] * w + j0;
#pragma unroll
      for (int v = 0; v < VEC; ++v) in[ii][v] = j0 + 32 * v < w ? u[32 * v] : 0.0f;
    }
  }
  for (int jj = 0; jj < m; jj += 4) {
    float s[4][VEC];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int v = 0; v < VEC; ++v) s[k][v] = 0.0f;
#pragma unroll
    for (int ii = 0; ii < MAXM; ++ii) {
      if (ii < m) {
        const float4 q = *reinterpret_cast<const float4*>(Qs + ii * MAXM + jj);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          s[0][v] = fmaf(q.x, in[ii][v], s[0][v]);
          s[1][v] = fmaf(q.y, in[ii][v], s[1][v]);
          s[2][v] = fmaf(q.z, in[ii][v], s[2][v]);
          s[3][v] = fmaf(q.w, in[ii][v], s[3][v]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (jj + k < m) {
        float* u = U + (int64_t)ss[jj + k] * w + j0;
#pragma unroll
        for (int v = 0; v < VEC; ++v)
          if (j0 + 32 * v < w) u[32 * v] = s[k][v];
      }
  }
}

// The same for clusters of more inputs than registers hold, through shared memory.
__global__ void rowfwt_kernel(Geo g, const int32_t* lvl, int w, float* U) {
  __shared__ float in[kMaxIn][kColTile];
  __shared__ float Qs[kMaxIn * kMaxIn];
  const int c = lvl[blockIdx.x];
  const int j0 = blockIdx.y * kColTile;
  const int cols = min(kColTile, w - j0);
  const int m = g.nin[c];
  const int32_t* sl = g.slots + g.slot_off[c];
  const float* Q = g.Q + g.qoff[c];
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) Qs[e] = Q[e];
  for (int e = threadIdx.x; e < m * kColTile; e += blockDim.x) {
    const int ii = e / kColTile, j = e - ii * kColTile;
    in[ii][j] = j < cols ? U[(int64_t)sl[ii] * w + j0 + j] : 0.0f;
  }
  __syncthreads();
  const int j = threadIdx.x % kColTile;
  for (int jj = threadIdx.x / kColTile; jj < m; jj += blockDim.x / kColTile) {
    float s = 0.0f;
    for (int ii = 0; ii < m; ++ii) s = fmaf(Qs[ii * m + jj], in[ii][j], s);
    if (j < cols) U[(int64_t)sl[jj] * w + j0 + j] = s;
  }
}

// In-place column transform of an N x m matrix G (row-major): G[r,:] <- G[r,:] Q.
__global__ void colfwt_rows_kernel(int64_t n, int m, const float* Q, float* G) {
  __shared__ float Qs[kMaxIn * kMaxIn];
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) Qs[e] = Q[e];
  __syncthreads();
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= n) return;
  float in[kMaxIn];
  for (int ii = 0; ii < m; ++ii) in[ii] = G[r * m + ii];
  for (int jj = 0; jj < m; ++jj) {
    float s = 0.0f;
    for (int ii = 0; ii < m; ++ii) s = fmaf(in[ii], Qs[ii * m + jj], s);
    G[r * m + jj] = s;
  }
}

// Extraction: entry e = block (a, b): staging[off + i*nb + j] = Src[rowslot[boff[a]+i], col[j]]
// with col[j] = colmap[cm_off[e] + j] - q0; bmax[k] = max |entry|.  One warp per entry.
struct Ext {
  const int32_t* a;
  const int32_t* b;
  const int64_t* off;   // staging offset
  const int32_t* k;     // upper-triangle block id (for bmax)
  const int32_t* cm;    // column map base index of each entry into colmap
};

__global__ void extract_kernel(Ext ex, int64_t nent, const int32_t* bsize, const int64_t* boff,
                               const int32_t* rowslot, const int32_t* colmap, int64_t q0, const float* Src,
                               int64_t ld, float* staging, float* bmax) {
  const int lane = threadIdx.x & 31;
  const int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (e >= nent) return;
  const int a = ex.a[e], b = ex.b[e];
  const int na = bsize[a], nb = bsize[b];
  const int32_t* cm = colmap + ex.cm[e];
  float* dst = staging + ex.off[e];
  float mx = 0.0f;
  for (int t = lane; t < na * nb; t += 32) {
    const int i = t / nb, j = t - i * nb;
    const float v = Src[(int64_t)rowslot[boff[a] + i] * ld + (cm[j] - q0)];
    dst[t] = v;
    mx = fmaxf(mx, fabsf(v));
  }
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) bmax[ex.k[e]] = mx;
}

// U[:, cols] -> S (N x m, row-major)
__global__ void gather_cols_kernel(int64_t n, int m, const int32_t* cols, int64_t q0, const float* U, int w,
                                   float* S) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * m) return;
  const int64_t r = t / m;
  const int j = (int)(t - r * m);
  S[t] = U[r * w + (cols[j] - q0)];
}

// concatenate two N x m0 / N x m1 row-major blocks into G (N x (m0+m1))
__global__ void concat_kernel(int64_t n, int m0, const float* A, int m1, const float* B, float* G) {
  const int m = m0 + m1;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * m) return;
  const int64_t r = t / m;
  const int j = (int)(t - r * m);
  G[t] = j < m0 ? A[r * m0 + j] : B[r * m1 + (j - m0)];
}

// Final values: block (a, b) of the kept pattern from the staged block of the pair, the
// nugget on the diagonal, entries below tau set to zero.
__global__ void assemble_kernel(int64_t nblk, const int32_t* brow, const int32_t* bcol, const int64_t* voff,
                                const int64_t* src_off, const int32_t* bsize, const float* staging, double nugget,
                                double tau, double* out) {
  const int lane = threadIdx.x & 31;
  const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (k >= nblk) return;
  const int a = brow[k], b = bcol[k];
  const int na = bsize[a], nb = bsize[b];
  const float* s = staging + src_off[k];
  double* o = out + voff[k];
  for (int t = lane; t < na * nb; t += 32) {
    const int i = t / nb, j = t - i * nb;
    double v = a <= b ? (double)s[t] : (double)s[j * na + i];  // staged block is (min, max)
    if (a == b && i == j) v += nugget;
    o[t] = fabs(v) < tau ? 0.0 : v;
  }
}

template <typename T>
static s_status dmalloc(T** p, size_t count) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * std::max<size_t>(count, 1));
  if (e != cudaSuccess) return cuda_error(e, "cudaMalloc(build values)");
  return S_OK;
}

template <typename T>
static s_status upload(T** p, const std::vector<T>& v) {
  s_status st = dmalloc(p, v.size());
  if (st) return st;
  if (!v.empty()) SF_CUDA(cudaMemcpy(*p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return S_OK;
}

struct Frees {
  std::vector<void*> ptrs;
  void add(void* p) { ptrs.push_back(p); }
  ~Frees() {
    for (void* p : ptrs) cudaFree(p);
  }
};

}  // namespace sf

using namespace sf;

s_build_t::~s_build_t() { cudaFree(dvals); }

// Values of the kernel (deriv = false) or of its ell-derivative (deriv = true).  Without a
// given pattern the kept pattern is decided by tau and returned in *pattern with the values
// held by the builder; with a given pattern (a sub-pattern of the eta pattern) the values on
// it are written to `out` (no threshold, no nugget).
static s_status values_impl(s_build b, double nu, double ell, double kscale, double nugget, double tau, bool deriv,
                            const s_pattern_t* given, double* out, s_pattern* pattern) {
  int p;
  if (std::fabs(nu - 0.5) < 1e-12) p = 0;
  else if (std::fabs(nu - 1.5) < 1e-12) p = 1;
  else if (std::fabs(nu - 2.5) < 1e-12) p = 2;
  else return set_error(S_ERR_ARG, "s_build_values: nu must be 0.5, 1.5 or 2.5");
  if (!(ell > 0.0)) return set_error(S_ERR_ARG, "s_build_values: ell must be positive");
  if (deriv) p += 3;
  const int64_t n = b->n;
  const int nc = (int)b->cl.size();
  for (const auto& c : b->cl)
    if (c.nin > kMaxIn) return set_error(S_ERR_ARG, "s_build_values: a cluster has more than 64 inputs");
  Frees fr;
  s_status st;
  // ---- geometry and transforms on the device ----------------------------------------
  std::vector<float> xf((size_t)n * 3, 0.0f);
  for (int64_t i = 0; i < n; ++i)
    for (int a = 0; a < b->d; ++a) xf[i * 3 + a] = (float)b->points[b->perm[i] * b->d + a];
  std::vector<int64_t> qoff(nc + 1, 0);
  for (int c = 0; c < nc; ++c) qoff[c + 1] = qoff[c] + (int64_t)b->cl[c].nin * b->cl[c].nin;
  std::vector<float> qf(qoff[nc]);
  std::vector<int32_t> nin(nc), ns(nc);
  for (int c = 0; c < nc; ++c) {
    for (size_t t = 0; t < b->cl[c].Q.size(); ++t) qf[qoff[c] + t] = (float)b->cl[c].Q[t];
    nin[c] = b->cl[c].nin;
    ns[c] = b->cl[c].ns;
  }
  Geo g{};
  float *dx, *dq;
  int64_t *dqoff, *dslot_off, *dboff;
  int32_t *dslots, *dnin, *dns, *drowslot, *dbsize;
  if ((st = upload(&dx, xf)) || (st = upload(&dq, qf)) || (st = upload(&dqoff, qoff)) ||
      (st = upload(&dslots, b->slots)) || (st = upload(&dslot_off, b->slot_off)) || (st = upload(&dnin, nin)) ||
      (st = upload(&dns, ns)) || (st = upload(&drowslot, b->rowslot)) || (st = upload(&dboff, b->block_offset)) ||
      (st = upload(&dbsize, b->bsize)))
    return st;
  for (void* q : {(void*)dx, (void*)dq, (void*)dqoff, (void*)dslots, (void*)dslot_off, (void*)dnin, (void*)dns,
                  (void*)drowslot, (void*)dboff, (void*)dbsize})
    fr.add(q);
  g.x = dx;
  g.Q = dq;
  g.qoff = dqoff;
  g.slots = dslots;
  g.slot_off = dslot_off;
  g.nin = dnin;
  g.ns = dns;
  // ---- upper-triangle block list (a <= b) and its staging offsets ---------------------
  // uid[k]: id of block k's unordered pair among the blocks (a, b), a <= b (-1: the pattern holds
  // (b, a) without (a, b)).  Rows are visited in order, so the mirrored blocks (b, a) of a row b
  // come up in that row's own order: one cursor per row, no searches.
  const std::vector<int64_t>& rp = b->rowptr;
  const std::vector<int32_t>& ci = b->colidx;
  const int64_t nb_all = (int64_t)ci.size();
  std::vector<int32_t> uid(nb_all, -1);
  std::vector<int64_t> ut_off;
  ut_off.reserve((size_t)(nb_all + nc) / 2 + 1);
  int64_t nut = 0, stage_total = 0;
  {
    std::vector<int64_t> cur(rp.begin(), rp.end() - 1);
    for (int a = 0; a < nc; ++a)
      for (int64_t k = std::lower_bound(ci.data() + rp[a], ci.data() + rp[a + 1], a) - ci.data(); k < rp[a + 1]; ++k) {
        const int c = ci[k];
        uid[k] = (int32_t)nut;
        if (c > a) {
          int64_t& q = cur[c];
          while (q < rp[c + 1] && ci[q] < a) ++q;
          if (q < rp[c + 1] && ci[q] == a) uid[q++] = (int32_t)nut;
        }
        ++nut;
        ut_off.push_back(stage_total);
        stage_total += (int64_t)b->bsize[a] * b->bsize[c];
      }
  }
  // column map of a cluster: its coordinate slots (root: scaling then samplets); behind it the
  // identity, the map of the clusters above the chunks (their columns are those of G)
  std::vector<int64_t> cm_base(nc);
  std::vector<int32_t> colmap;
  for (int c = 0; c < nc; ++c) {
    cm_base[c] = (int64_t)colmap.size();
    const int32_t* sl = b->slots.data() + b->slot_off[c];
    const int base = c == 0 ? 0 : b->cl[c].ns;
    for (int j = 0; j < b->bsize[c]; ++j) colmap.push_back(sl[base + j]);
  }
  const int64_t ident = (int64_t)colmap.size();
  for (int j = 0; j < kMaxIn; ++j) colmap.push_back(j);
  float *dstage, *dbmax;
  int32_t* dcolmap;
  if ((st = dmalloc(&dstage, stage_total))) return st;
  fr.add(dstage);
  if ((st = dmalloc(&dbmax, nut))) return st;
  fr.add(dbmax);
  if ((st = upload(&dcolmap, colmap))) return st;
  fr.add(dcolmap);
  SF_CUDA(cudaMemset(dbmax, 0, sizeof(float) * std::max<int64_t>(nut, 1)));
  // ---- chunks: maximal clusters with at most kChunk points ------------------------------
  std::vector<int32_t> chunks;  // chunk roots in left-to-right order
  {
    std::vector<int32_t> st2{0};
    while (!st2.empty()) {
      int c = st2.back();
      st2.pop_back();
      if (b->cl[c].hi - b->cl[c].lo <= kChunk || b->cl[c].son[0] < 0) {
        chunks.push_back(c);
      } else {
        st2.push_back(b->cl[c].son[1]);
        st2.push_back(b->cl[c].son[0]);
      }
    }
  }
  int wmax = 0;
  for (int c : chunks) wmax = std::max<int>(wmax, (int)(b->cl[c].hi - b->cl[c].lo));
  float* dU;
  if ((st = dmalloc(&dU, (size_t)n * wmax))) return st;
  fr.add(dU);
  // Every list that the chunk loop needs, uploaded once: the subtree of each chunk (deepest level
  // first) and the extraction entries of each chunk and of each cluster above.  Per column cluster
  // bb the entries are the blocks (a, bb), a <= bb.
  struct Range {
    int64_t b = 0, e = 0;
  };
  std::vector<int32_t> sub_all, sub_lvl;       // clusters, level offsets (relative to the chunk's first)
  std::vector<Range> sub_at(chunks.size()), lvl_at(chunks.size()), ent_at(chunks.size()), up_at(nc);
  std::vector<int32_t> ea, eb, ek, ecm;
  std::vector<int64_t> eo;
  const size_t half_blocks = (size_t)nut;
  ea.reserve(half_blocks), eb.reserve(half_blocks), ek.reserve(half_blocks), ecm.reserve(half_blocks);
  eo.reserve(half_blocks);
  auto entries_of = [&](int bb, int64_t cm) {
    for (int64_t k = rp[bb]; k < rp[bb + 1] && ci[k] <= bb; ++k) {
      if (uid[k] < 0) continue;  // pattern not symmetric here: skip
      ea.push_back(ci[k]);
      eb.push_back(bb);
      eo.push_back(ut_off[uid[k]]);
      ek.push_back(uid[k]);
      ecm.push_back((int32_t)cm);
    }
  };
  std::vector<uint8_t> in_chunk(nc, 0);
  for (size_t q = 0; q < chunks.size(); ++q) {
    const int gch = chunks[q];
    std::vector<std::vector<int32_t>> sl(b->depth + 1);
    std::vector<int32_t> st3{gch}, members;
    while (!st3.empty()) {
      int c = st3.back();
      st3.pop_back();
      members.push_back(c);
      in_chunk[c] = 1;
      sl[b->cl[c].level].push_back(c);
      if (b->cl[c].son[0] >= 0) {
        st3.push_back(b->cl[c].son[0]);
        st3.push_back(b->cl[c].son[1]);
      }
    }
    sub_at[q].b = (int64_t)sub_all.size();
    lvl_at[q].b = (int64_t)sub_lvl.size();
    sub_lvl.push_back(0);
    for (int L = b->depth; L >= b->cl[gch].level; --L) {
      sub_all.insert(sub_all.end(), sl[L].begin(), sl[L].end());
      sub_lvl.push_back((int32_t)((int64_t)sub_all.size() - sub_at[q].b));
    }
    sub_at[q].e = (int64_t)sub_all.size();
    lvl_at[q].e = (int64_t)sub_lvl.size();
    ent_at[q].b = (int64_t)ea.size();
    for (int c : members)
      if (b->bsize[c] > 0) entries_of(c, cm_base[c]);
    ent_at[q].e = (int64_t)ea.size();
  }
  for (int c = 0; c < nc; ++c)
    if (!in_chunk[c]) {
      up_at[c].b = (int64_t)ea.size();
      if (b->bsize[c] > 0) entries_of(c, ident + (c == 0 ? 0 : b->cl[c].ns));
      up_at[c].e = (int64_t)ea.size();
    }
  // levels of the row tree, deepest first
  std::vector<std::vector<int32_t>> bylev(b->depth + 1);
  for (int c = 0; c < nc; ++c) bylev[b->cl[c].level].push_back(c);
  std::vector<int32_t> lvl_flat, lvl_off{0};
  std::vector<int> lvl_m;  // widest transform of each level
  for (int L = b->depth; L >= 0; --L) {
    lvl_flat.insert(lvl_flat.end(), bylev[L].begin(), bylev[L].end());
    lvl_off.push_back((int32_t)lvl_flat.size());
    int mm = 0;
    for (int32_t c : bylev[L]) mm = std::max(mm, b->cl[c].nin);
    lvl_m.push_back(mm);
  }
  int32_t *dlvl, *dsub, *dsublvl, *da, *db, *dk, *dcm;
  int64_t* dof;
  for (auto up : {std::make_pair(&dlvl, &lvl_flat), std::make_pair(&dsub, &sub_all), std::make_pair(&dsublvl, &sub_lvl),
                  std::make_pair(&da, &ea), std::make_pair(&db, &eb), std::make_pair(&dk, &ek), std::make_pair(&dcm, &ecm)}) {
    if ((st = upload(up.first, *up.second))) return st;
    fr.add(*up.first);
  }
  if ((st = upload(&dof, eo))) return st;
  fr.add(dof);
  int maxm = 1, maxns = 1;
  for (const auto& c : b->cl) {
    maxm = std::max(maxm, c.nin);
    maxns = std::max(maxns, c.ns);
  }
  const int mp = (maxm + 1) & ~1;
  const size_t smem = sizeof(float) * ((size_t)kRowTile * wmax + 8 * (size_t)(maxm * mp + mp));
  SF_CUDA(cudaFuncSetAttribute(eval_colfwt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // Scaling columns of finished clusters, waiting for their sibling: (cluster, N x ns buffer).  The
  // buffers are reused (at most one per level waits; everything is on one stream), as is G.
  std::vector<std::pair<int32_t, float*>> stack;
  std::vector<float*> spare;
  auto take = [&](float** out) -> s_status {
    if (!spare.empty()) {
      *out = spare.back();
      spare.pop_back();
      return S_OK;
    }
    s_status s2 = dmalloc(out, (size_t)n * maxns);
    if (!s2) fr.add(*out);
    return s2;
  };
  float* Gm = nullptr;
  if (chunks.size() > 1) {
    if ((st = dmalloc(&Gm, (size_t)n * maxm))) return st;
    fr.add(Gm);
  }
  auto run_extract = [&](const Range& r, int64_t q0, const float* src, int64_t ld) -> s_status {
    const int64_t ne = r.e - r.b;
    if (ne == 0) return S_OK;
    Ext ex{da + r.b, db + r.b, dof + r.b, dk + r.b, dcm + r.b};
    extract_kernel<<<(unsigned)((ne * 32 + 255) / 256), 256>>>(ex, ne, dbsize, dboff, drowslot, dcolmap, q0, src, ld,
                                                             dstage, dbmax);
    SF_CUDA(cudaGetLastError());
    return S_OK;
  };
  // the scaling columns of cluster c: `cols` of src (ld columns, first column q0)
  auto keep_scaling = [&](int c, const int32_t* dcols, int64_t q0, const float* src, int ld) -> s_status {
    float* S;
    s_status s2 = take(&S);
    if (s2) return s2;
    const int nsc = b->cl[c].ns;
    if (nsc > 0)
      gather_cols_kernel<<<(unsigned)((n * nsc + 255) / 256), 256>>>(n, nsc, dcols, q0, src, ld, S);
    SF_CUDA(cudaGetLastError());
    stack.push_back({c, S});
    return S_OK;
  };
  for (size_t q = 0; q < chunks.size(); ++q) {
    const int gch = chunks[q];
    const BCluster& G = b->cl[gch];
    const int64_t q0 = G.lo;
    const int w = (int)(G.hi - G.lo);
    eval_colfwt_kernel<<<(unsigned)((n + kRowTile - 1) / kRowTile), 256, smem>>>(
        g, n, q0, w, dsub + sub_at[q].b, dsublvl + lvl_at[q].b, (int)(lvl_at[q].e - lvl_at[q].b) - 1, p, (float)(1.0 / ell),
        (float)kscale, maxm, dU);
    SF_CUDA(cudaGetLastError());
    for (int L = 0; L < (int)lvl_off.size() - 1; ++L) {
      const int cnt = lvl_off[L + 1] - lvl_off[L];
      if (!cnt) continue;
      const int32_t* lv = dlvl + lvl_off[L];
      // a CTA per cluster with a warp per 128 (64) columns, the registers for the level's widest cluster
      const int warps = (w + 127) / 128, warps2 = std::min(8, (w + 63) / 64);
      if (lvl_m[L] <= 12) rowfwt_reg_kernel<12, 4><<<cnt, 32 * warps>>>(g, lv, w, dU);
      else if (lvl_m[L] <= 20) rowfwt_reg_kernel<20, 4><<<cnt, 32 * warps>>>(g, lv, w, dU);
      else if (lvl_m[L] <= 40)
        rowfwt_reg_kernel<40, 2><<<dim3(cnt, (w + 64 * warps2 - 1) / (64 * warps2)), 32 * warps2>>>(g, lv, w, dU);
      else rowfwt_kernel<<<dim3(cnt, (w + kColTile - 1) / kColTile), 256>>>(g, lv, w, dU);
    }
    SF_CUDA(cudaGetLastError());
    if ((st = run_extract(ent_at[q], q0, dU, w))) return st;
    if (gch == 0) break;  // the whole tree was one chunk
    if ((st = keep_scaling(gch, dslots + b->slot_off[gch], q0, dU, w))) return st;
    // combine finished siblings upwards
    while (stack.size() >= 2) {
      auto s1 = stack[stack.size() - 1], s0 = stack[stack.size() - 2];
      const int par = b->cl[s0.first].parent;
      if (par < 0 || par != b->cl[s1.first].parent || b->cl[par].son[0] != s0.first) break;
      stack.pop_back();
      stack.pop_back();
      const int m = b->cl[par].nin;
      concat_kernel<<<(unsigned)((n * m + 255) / 256), 256>>>(n, b->cl[s0.first].ns, s0.second, b->cl[s1.first].ns,
                                                              s1.second, Gm);
      colfwt_rows_kernel<<<(unsigned)((n + 127) / 128), 128>>>(n, m, dq + qoff[par], Gm);
      SF_CUDA(cudaGetLastError());
      spare.push_back(s0.second);
      spare.push_back(s1.second);
      if ((st = run_extract(up_at[par], 0, Gm, m))) return st;
      if (par == 0) break;
      if ((st = keep_scaling(par, dcolmap + ident, 0, Gm, m))) return st;  // the first ns columns of G
    }
  }
  SF_CUDA(cudaDeviceSynchronize());
  // ---- kept pattern (decided per unordered pair), or the given one ----------------------
  std::vector<float> bmax(nut);
  SF_CUDA(cudaMemcpy(bmax.data(), dbmax, sizeof(float) * nut, cudaMemcpyDeviceToHost));
  std::vector<int64_t> krp(nc + 1, 0);
  std::vector<int32_t> kci;
  std::vector<int64_t> ksrc;
  if (given) {
    if (given->d.nc != nc) return set_error(S_ERR_MISMATCH, "s_build_values_dell: pattern from another tree");
    kci.reserve(given->colidx.size());
    ksrc.reserve(given->colidx.size());
    for (int a = 0; a < nc; ++a) {
      int64_t q = rp[a];  // both rows are sorted
      for (int64_t k = given->rowptr[a]; k < given->rowptr[a + 1]; ++k) {
        const int c = given->colidx[k];
        while (q < rp[a + 1] && ci[q] < c) ++q;
        int64_t u = q < rp[a + 1] && ci[q] == c ? uid[q] : -1;
        if (u < 0 && c < a) {  // held as (c, a) only
          const int32_t* end = ci.data() + rp[c + 1];
          const int32_t* pos = std::lower_bound(ci.data() + rp[c], end, a);
          if (pos != end && *pos == a) u = uid[pos - ci.data()];
        }
        if (u < 0) return set_error(S_ERR_PATTERN, "s_build_values_dell: block outside the eta pattern");
        kci.push_back(c);
        ksrc.push_back(ut_off[u]);
      }
      krp[a + 1] = (int64_t)kci.size();
    }
  } else {
    kci.reserve(nb_all);
    ksrc.reserve(nb_all);
    for (int a = 0; a < nc; ++a) {
      for (int64_t k = rp[a]; k < rp[a + 1]; ++k) {
        const int c = ci[k];
        const int64_t u = uid[k];
        if (u < 0) continue;
        if (a == c || (double)bmax[u] >= tau) {
          kci.push_back(c);
          ksrc.push_back(ut_off[u]);
        }
      }
      krp[a + 1] = (int64_t)kci.size();
    }
  }
  s_pattern pat = nullptr;
  const s_pattern_t* tgt = given;
  if (!given) {
    if ((st = s_pattern_create(nc, b->block_offset.data(), b->level.data(), krp.data(), kci.data(), &pat))) return st;
    tgt = pat;
  }
  const int64_t nnz = tgt->d.nnz;
  double* vals = out;
  if (!given) {
    cudaError_t e = cudaMalloc(&vals, sizeof(double) * std::max<int64_t>(nnz, 1));
    if (e != cudaSuccess) {
      s_pattern_destroy(pat);
      return cuda_error(e, "cudaMalloc(values)");
    }
  }
  int64_t* dsrc;
  if ((st = upload(&dsrc, ksrc))) {
    if (!given) {
      s_pattern_destroy(pat);
      cudaFree(vals);
    }
    return st;
  }
  fr.add(dsrc);
  const int64_t nk = (int64_t)kci.size();
  if (nk)
    assemble_kernel<<<(unsigned)((nk * 32 + 255) / 256), 256>>>(nk, tgt->d.brow, tgt->d.colidx, tgt->d.voff, dsrc,
                                                              dbsize, dstage, given ? 0.0 : nugget,
                                                              given ? 0.0 : tau, vals);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    if (!given) {
      s_pattern_destroy(pat);
      cudaFree(vals);
    }
    return cuda_error(e, "assemble_kernel");
  }
  if (!given) {
    *pattern = pat;
    b->dvals = vals;
    b->nvals = nnz;
  }
  return S_OK;
}

extern "C" s_status s_build_values(s_build b, double nu, double ell, double kscale, double nugget, double tau,
                                   s_pattern* pattern) {
  if (!b || !pattern) return set_error(S_ERR_ARG, "s_build_values: NULL argument");
  *pattern = nullptr;
  cudaFree(b->dvals);
  b->dvals = nullptr;
  b->nvals = 0;
  return values_impl(b, nu, ell, kscale, nugget, tau, false, nullptr, nullptr, pattern);
}

// y = (kscale K + nugget I) v with every kernel entry evaluated (no compression): one thread
// per row, columns streamed through shared memory 1024 at a time; each tile's terms summed in
// float, the tiles in double.
constexpr int kMvTile = 1024;
__global__ void __launch_bounds__(256) kmatvec_kernel(const float* __restrict__ x, int64_t n, int p, float inv_ell,
                                                      float scale, const float* __restrict__ v, double* __restrict__ y) {
  __shared__ float sx[kMvTile][3];
  __shared__ float sv[kMvTile];
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool row = i < n;
  const float xi0 = row ? x[i * 3] : 0.f, xi1 = row ? x[i * 3 + 1] : 0.f, xi2 = row ? x[i * 3 + 2] : 0.f;
  double acc = 0.0;
  for (int64_t j0 = 0; j0 < n; j0 += kMvTile) {
    const int cnt = (int)(n - j0 < kMvTile ? n - j0 : (int64_t)kMvTile);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
      sx[t][0] = x[(j0 + t) * 3];
      sx[t][1] = x[(j0 + t) * 3 + 1];
      sx[t][2] = x[(j0 + t) * 3 + 2];
      sv[t] = v[j0 + t];
    }
    __syncthreads();
    float part = 0.f;
    for (int t = 0; t < cnt; ++t) {
      const float d0 = xi0 - sx[t][0], d1 = xi1 - sx[t][1], d2 = xi2 - sx[t][2];
      const float r = sqrtf(fmaf(d0, d0, fmaf(d1, d1, d2 * d2)));
      part = fmaf(matern(r, p, inv_ell, scale), sv[t], part);
    }
    acc += (double)part;
  }
  if (row) y[i] = acc;
}

extern "C" s_status s_build_kernel_matvec(s_build b, double nu, double ell, double kscale, double nugget,
                                          const double* v, double* y) {
  if (!b || !v || !y) return set_error(S_ERR_ARG, "s_build_kernel_matvec: NULL argument");
  int p;
  if (std::fabs(nu - 0.5) < 1e-12) p = 0;
  else if (std::fabs(nu - 1.5) < 1e-12) p = 1;
  else if (std::fabs(nu - 2.5) < 1e-12) p = 2;
  else return set_error(S_ERR_ARG, "s_build_kernel_matvec: nu must be 0.5, 1.5 or 2.5");
  if (!(ell > 0.0)) return set_error(S_ERR_ARG, "s_build_kernel_matvec: ell must be positive");
  const int64_t n = b->n;
  std::vector<float> xf((size_t)n * 3, 0.0f), vf(n);
  for (int64_t i = 0; i < n; ++i) {
    for (int a = 0; a < b->d; ++a) xf[i * 3 + a] = (float)b->points[i * b->d + a];
    vf[i] = (float)v[i];
  }
  Frees fr;
  s_status st;
  float *dx, *dv;
  double* dy;
  if ((st = upload(&dx, xf)) || (st = upload(&dv, vf)) || (st = dmalloc(&dy, (size_t)n))) return st;
  fr.add(dx);
  fr.add(dv);
  fr.add(dy);
  kmatvec_kernel<<<(unsigned)((n + 255) / 256), 256>>>(dx, n, p, (float)(1.0 / ell), (float)kscale, dv, dy);
  SF_CUDA(cudaGetLastError());
  SF_CUDA(cudaMemcpy(y, dy, sizeof(double) * n, cudaMemcpyDeviceToHost));
  for (int64_t i = 0; i < n; ++i) y[i] += nugget * v[i];
  return S_OK;
}

extern "C" s_status s_build_values_dell(s_build b, double nu, double ell, double kscale, s_pattern on, double* out) {
  if (!b || !on || (!out && on->d.nnz > 0)) return set_error(S_ERR_ARG, "s_build_values_dell: NULL argument");
  return values_impl(b, nu, ell, kscale, 0.0, 0.0, true, on, out, nullptr);
}

extern "C" s_status s_build_take_values(s_build b, double* dst, void* stream) {
  if (!b || (!dst && b->nvals > 0)) return set_error(S_ERR_ARG, "s_build_take_values: NULL argument");
  if (!b->dvals) return set_error(S_ERR_ARG, "s_build_take_values: no values (call s_build_values first)");
  if (b->nvals) SF_CUDA(cudaMemcpyAsync(dst, b->dvals, sizeof(double) * b->nvals, cudaMemcpyDeviceToDevice,
                                        (cudaStream_t)stream));
  SF_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
  cudaFree(b->dvals);
  b->dvals = nullptr;
  b->nvals = 0;
  return S_OK;
}
