// Float masked product C = P_{S_C}(op(X) op(Y)) (Eq. (product), Sec. 4.1) with both operands
// packed for the multiply-add loop.
//
// Operand layout ("t pairs"): for the X side the slice op(X)(nu, lambda) has a row per row of
// nu, for the Y side op(Y)(lambda, nu') a row per column of nu', t running over lambda's
// samplets.  A pre-pass (nt_prepare_kernel) writes each block, transposed as needed, into
// plan-owned scratch as panels of at most 20 rows, a panel as [t / 2][row][t % 2]: t padded to
// even with zeros, every block on a 16-byte boundary.  A range of t that starts at a multiple of
// kNtKC is then one contiguous, aligned run for all rows of an output tile, and a lane finds its
// MR rows' pairs side by side at constant offsets.  With B = A declared symmetric one copy
// serves both sides.  The pre-pass moves 8 bytes an entry once where the product reads each
// operand entry some 20 to 300 times.
//
// Lists: the matching lambda blocks of every block of S_C (where both operands' slices start, the
// t extent) are written once by nt_list_kernel, one warp per block, and kept by the plan while there
// is memory to spare (kNtListMax); beyond that every product lists and multiplies range after
// range of blocks through a workspace (kNtListWork).  Intersecting inside the product kernel cost more
// than the products of narrow blocks: in the plane the lists of a tile are 300 entries long for
// 60 matches.
//
// Work decomposition: one warp owns one output tile (at most 20 x 20 entries of one block of
// S_C) for the whole lambda sum.  The tile is cut into a GR x GC grid of MR x MC micro-tiles,
// GR = 2 for tiles of at most 10 rows and 4 beyond (GC likewise), one lane per micro-tile, and
// the 32 / (GR GC) lane groups take consecutive lambda blocks of the tile's list (split-K): 8
// blocks at once for tiles up to 10 x 10, 2 for tiles beyond 10 both ways.  The control of a
// step is paid once for all its blocks, so narrow blocks, whose products are only 7 to 30
// multiply-add instructions, run 8 to a step.  A lane's step over a pair of t is MR + MC 8-byte
// shared loads and MR MC packed multiply-adds (fma.rn.f32x2 over the two values of t).  What
// bounds it: shared memory delivers 128 bytes per clock and SM to registers, i.e.
// 8 (MR + MC) 32 / 128 clocks for a pair of t against MR MC / 2 clocks of the float pipes, 62 %
// of the float peak for 5 x 5 micro-tiles (a loop of nothing else measured 42 to 49 TFLOP/s,
// packed or not; packing halves the issue slots of the multiply-adds, which the control
// instructions need); the narrow tiles are bound by latency at 4 warps a scheduler.
//
// Staging: each lane group copies its own block with 16-byte cp.async (14 instructions a step
// for 8 blocks of 10 x 10).  One bulk copy per operand and block took longer on narrow blocks
// (a bulk copy issues from uniform registers, so a warp sends its 16 copies one lane at a time):
// 41.5 against 37.6 ms for the three products of a gradient step at N = 6000 in space, q = 2.
//
// Sums: even and odd t are two float partials per entry; after the first step, then every 4 (8 of
// wide tiles), they are added and folded into the running sum with an error-free two-sum,
// the rounding error carried in the partial.  The lists run from coarse to fine clusters, so
// the first step holds the largest terms: folded at once, it does not make the small terms that
// follow round at its size.  At the end the groups' sums are combined the same way in group
// order.  The order is fixed (deterministic).  Within a block t runs downwards, so a cluster's
// coarsest samplets, the largest terms of the dominant entries, are added last and round once.
// Error against 64 bits, geometric mean over 8 matrices of 500 to 9900 points: 0.2e-7 to 1.4e-7
// in the four families with 20- and 10-wide blocks.  Folding narrow tiles only every 16 steps is
// 0.8 % faster, but leaves the float square root at N = 2000 in space, whose factors are near the
// identity, 2.6e-7 off instead of 1.1e-7; t upwards is 0.4 % faster and takes the error at
// N = 5000 in the plane from 1.7e-8 to 6.8e-8.
//
// Measured (in brackets a kernel with K-major slices that intersects the lists itself, one half-warp
// per lambda block): N = 50000 in the plane, 10-wide blocks, B not symmetric 3.98 ms (9.27); N = 65536 in
// space, 20-wide blocks, B = A symmetric 30.5 ms, 37.5 TFLOP/s (39.1); N = 1000 in the plane 60 us
// (192); N = 500 in space, 20-wide 43 us (45 symmetric, 56 not); three products of a gradient
// step, N = 6000, 10-wide blocks 35.6 ms (107.6).
#include <algorithm>
#include <cstring>
#include <new>

#include "common.cuh"

namespace sf {
namespace {

constexpr int kNtWarps = 4;
constexpr int kNtKC = 20;        // largest t extent of a listed piece
constexpr int kNtBuf = 1632;     // floats of a stage buffer: 2 x 20x20x2 or 8 x 10x10x2 slices, and room to
                                 // start the 8 slots 12 banks apart (conflict-free 8-byte loads)
constexpr int kNtSlack = 64;     // a micro-tile reads up to 5 rows' pairs beyond its operand's last
constexpr int kNtAhead = 6;      // tiles per resident warp from which warps take tiles ahead (see the kernel)
constexpr size_t kNtSmem = sizeof(float) * (kNtWarps * 2 * kNtBuf + kNtSlack);
// Bytes of lists a plan keeps, and of the workspace beyond that.  Lists are many times the size of a
// matrix of narrow blocks (2.8 GB beside 87 MB at N = 6000 in space), so they are kept only while
// they leave half of the device's memory free, and the workspace is at most 1/512 of what is
// free: 256 plans of a batch (611 GB of lists) stay together on one GPU.  Range by range a product
// lists again and drains between ranges: N = 65536 in space, 20-wide 30.9 -> 33.7 ms, N = 250000 in the
// plane, 10-wide 19.9 -> 32.1 ms (39.1 with 64 MiB of workspace, 29.0 with 1 GiB).  4 GiB hold the
// lists of 2.7e8 block triples; beyond, N = 10^6 in the plane (7.9 GB) takes 139 ms, 85 with its lists
// kept, N = 10^5 in space (11.2 GB) 321 and 271 ms.
constexpr int64_t kNtListMax = (int64_t)4 << 30;
constexpr int64_t kNtListWork = (int64_t)256 << 20;
constexpr int64_t kNtListLeast = (int64_t)1 << 20;

// Padded t extent of a slice over nl values of t.
__host__ __device__ __forceinline__ int nt_even(int nl) { return (nl + 1) & ~1; }

struct NtArgs {
  const float* X;        // packed operands
  const float* Y;
  const NtEntry* ent;    // lists of the launch's range, from entry `base` on
  int64_t base;
  const NtTile* tiles;   // the launch's tiles
  uint32_t ntiles;
  unsigned int* counter;
  float* C;
};

// What the listing kernel needs of a side: the lists of op(X)'s rows or op(Y)'s columns (lambda
// ids, block ids or nullptr: position) and the float offset of each packed block.
struct NtSide {
  const int64_t* ptr;
  const int32_t* idx;
  const int32_t* blk;
  const int64_t* off;
};

// Matching lambda blocks of the blocks k0 .. k1-1 of S_C in increasing lambda order, one warp per
// block: the entries of the shorter list, 32 at a time, are looked up in the longer one by
// binary search.  A lambda block wider than kNtKC gives one entry per piece of kNtKC values of t.
// FILL: writes the entries at ent[eptr[k] - base ..); else writes their number to cnt[k].
template <bool FILL>
__global__ void __launch_bounds__(256) nt_list_kernel(NtSide x, NtSide y, const int32_t* __restrict__ bsize,
                                                      const int32_t* __restrict__ c_brow,
                                                      const int32_t* __restrict__ c_col, int64_t k0, int64_t k1,
                                                      int32_t* __restrict__ cnt, const int64_t* __restrict__ eptr,
                                                      int64_t base, NtEntry* __restrict__ ent) {
  const int lane = threadIdx.x & 31;
  for (int64_t k = k0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5); k < k1;
       k += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int nu = c_brow[k], nup = c_col[k];
    const int px0 = (int)x.ptr[nu], nx = (int)x.ptr[nu + 1] - px0;
    const int py0 = (int)y.ptr[nup], ny = (int)y.ptr[nup + 1] - py0;
    const bool xs = nx <= ny;  // walk X's list, search Y's
    const int32_t* sidx = xs ? x.idx + px0 : y.idx + py0;
    const int32_t* lidx = xs ? y.idx + py0 : x.idx + px0;
    const int ns = xs ? nx : ny, nl = xs ? ny : nx;
    int lo0 = 0, total = 0;
    NtEntry* out = FILL ? ent + (eptr[k] - base) : nullptr;
    for (int i0 = 0; i0 < ns && lo0 < nl; i0 += 32) {
      const int i = i0 + lane;
      const int32_t v = i < ns ? __ldg(sidx + i) : INT32_MAX;
      int lo = lo0, hi = nl;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(lidx + mid) < v) lo = mid + 1;
        else hi = mid;
      }
      const bool hit = i < ns && lo < nl && __ldg(lidx + lo) == v;
      const int kp = hit ? nt_even(__ldg(bsize + v)) : 0;
      const int np = (kp + kNtKC - 1) / kNtKC;
      int incl = np;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
      }
      if (FILL && hit) {
        const int ix = px0 + (xs ? i : lo), iy = py0 + (xs ? lo : i);
        NtEntry en;
        en.xo = (uint32_t)(__ldg(x.off + (x.blk ? __ldg(x.blk + ix) : ix)) >> 2);
        en.yo = (uint32_t)(__ldg(y.off + (y.blk ? __ldg(y.blk + iy) : iy)) >> 2);
        en.kp = kp;
        for (int j = 0; j < np; ++j) {
          en.t0 = j * kNtKC;
          en.kc = min(kNtKC, kp - en.t0);
          out[total + incl - np + j] = en;
        }
      }
      total += __shfl_sync(0xffffffffu, incl, 31);
      lo0 = __shfl_sync(0xffffffffu, lo, 31);
    }
    if (!FILL && lane == 0) cnt[k] = total;
  }
}

// The tiles of every block of S_C, in block order: block k's tiles start at tptr[k].
__global__ void nt_tile_kernel(int64_t nb, const int32_t* __restrict__ bsize, const int32_t* __restrict__ c_brow,
                               const int32_t* __restrict__ c_col, const int64_t* __restrict__ c_voff,
                               const int64_t* __restrict__ tptr, const int64_t* __restrict__ eptr,
                               NtTile* __restrict__ tiles) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= nb) return;
  const int ni = bsize[c_brow[k]], nj = bsize[c_col[k]];
  NtTile* o = tiles + tptr[k];
  NtTile t;
  t.e0 = eptr[k];
  t.ne = (int32_t)(eptr[k + 1] - eptr[k]);
  t.nj = nj;
  for (int r0 = 0; r0 < ni; r0 += kTile)
    for (int c0 = 0; c0 < nj; c0 += kTile) {
      t.coff = c_voff[k] + (int64_t)r0 * nj + c0;
      t.r0 = (uint16_t)r0;
      t.c0 = (uint16_t)c0;
      t.th = (uint16_t)min(kTile, ni - r0);
      t.tw = (uint16_t)min(kTile, nj - c0);
      *o++ = t;
    }
}

// 16-byte asynchronous copy global -> shared: through L1 for the narrow tiles (GL = 4), whose
// neighbours re-read the same small slices soon (gradient step at N = 6000 in space 5 % faster), past
// L1 for the others (with it N = 65536 in space took 35.4 instead of 30.4 ms).
template <bool L1>
__device__ __forceinline__ void nt_cp16(uint32_t dst, const float* src) {
  if (L1) asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// n pieces of 16 bytes by the GL lanes of a group, CI a lane at a time with constant offsets.
template <int CI, int GL>
__device__ __forceinline__ void nt_copy(uint32_t dst, const float* src, int n, int gl) {
  dst += 16u * (uint32_t)gl;
  src += 4 * gl;
  for (int c = gl; c < n; c += CI * GL, dst += 16 * CI * GL, src += 4 * CI * GL) {
#pragma unroll
    for (int i = 0; i < CI; ++i)
      if (c + i * GL < n) nt_cp16<GL == 4>(dst + 16 * i * GL, src + 4 * i * GL);
  }
}

__device__ __forceinline__ void nt_fma2(unsigned long long& d, unsigned long long x, unsigned long long y) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(x), "l"(y));
}

// acc + p as an error-free two-sum: acc <- rounded sum, p <- its rounding error
__device__ __forceinline__ void nt_fold(float& acc, float& p) {
  const float s = acc + p;
  const float bp = s - acc;
  const float e = (acc - (s - bp)) + (p - bp);
  acc = s;
  p = e;
}

// the two partials of an entry added and folded; the error stays in the even partial
__device__ __forceinline__ void nt_fold2(float& acc, unsigned long long& p) {
  float v = __uint_as_float((unsigned int)p) + __uint_as_float((unsigned int)(p >> 32));
  nt_fold(acc, v);
  p = (unsigned long long)__float_as_uint(v);
}

__device__ __forceinline__ float2 nt_sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }

// One output tile of at most GR MR x GC MC entries.
template <int GR, int MR, int GC, int MC>
__device__ __forceinline__ void nt_tile(const NtArgs& a, const NtTile& tile, float* wbase, uint32_t wsmem, int lane) {
  constexpr int GL = GR * GC, S = 32 / GL, NQ = MR * MC, TW = GC * MC, NE = GR * MR * TW;
  // t extents up to KMAX fit S slots in a stage buffer, those up to kNtKC half as many
  constexpr int SLOT = kNtBuf / S, KMAX = S == 8 ? 10 : S == 4 ? 12 : kNtKC;
  // 16-byte pieces a lane copies of an X and of a Y slice of up to KMAX
  constexpr int CX = (GR * MR * KMAX / 4 + GL - 1) / GL, CY = (TW * KMAX / 4 + GL - 1) / GL;
  constexpr int FOLD = S == 2 ? 8 : 4;  // steps per two-sum fold: partials of 20 to 80 terms
  static_assert(S * ((NE + 1) & ~1) * 2 <= 2 * kNtBuf, "the group sums reuse the stage buffers");
  static_assert((GR * MR + TW) * KMAX <= SLOT && (GR * MR + TW) * kNtKC <= (S == 2 ? 1 : 2) * SLOT, "slot too small");
  const int g = lane / GL, gl = lane % GL, mr = gl / GC, mc = gl % GC;
  const int th = tile.th, tw = tile.tw, ne = tile.ne;
  float acc[NQ];
  unsigned long long p[NQ];
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    acc[i] = 0.0f;
    p[i] = 0ull;
  }
  const NtEntry* ep = a.ent + (tile.e0 - a.base);
  int folded = FOLD - 1, buf = 0, pos = 0;  // the first step is folded at once
  int cn = 0, ckc = 0, cxs = 0, cys = 0;  // the step in flight: blocks, this lane's t extent and slices
  NtEntry en = {};
  if (ne > 0) en = ep[min(g, ne - 1)];  // the group's block of the next step
  for (;;) {
    // ---- issue the next step into `buf`: each group copies its block's X slice, then its Y slice
    int nn = 0, nkc = 0, nxs = 0, nys = 0;
    if (pos < ne) {
      nn = min(S, ne - pos);
      const bool half = S > 2 && __any_sync(0xffffffffu, en.kc > KMAX);
      if (half) nn = min(nn, S / 2);
      nkc = g < nn ? (int)en.kc : 0;
      const int nx = (th * nkc + 3) >> 2, ny = (tw * nkc + 3) >> 2;  // 16-byte pieces
      nxs = buf * kNtBuf + g * (half ? 2 * SLOT : SLOT);
      nys = nxs + 4 * nx;
      nt_copy<CX, GL>(wsmem + 4u * (uint32_t)nxs,
                      a.X + ((int64_t)en.xo * 4 + ((int64_t)tile.r0 * en.kp + th * (int)en.t0)), nx, gl);
      nt_copy<CY, GL>(wsmem + 4u * (uint32_t)nys,
                      a.Y + ((int64_t)en.yo * 4 + ((int64_t)tile.c0 * en.kp + tw * (int)en.t0)), ny, gl);
      pos += nn;
      if (pos < ne) en = ep[min(pos + g, ne - 1)];  // arrives during this step's multiply-adds
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // ---- multiply the step in flight ---------------------------------------------------------
    if (cn > 0) {
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncwarp();
      // downwards: a cluster's first samplets are its coarsest, their terms the largest
      const float* xs = wbase + cxs + mr * (2 * MR) + ckc * th;
      const float* ys = wbase + cys + mc * (2 * MC) + ckc * tw;
#pragma unroll 2
      for (int t = ckc; t > 0; t -= 2) {
        xs -= 2 * th;
        ys -= 2 * tw;
        unsigned long long xv[MR];
#pragma unroll
        for (int i = 0; i < MR; ++i) xv[i] = reinterpret_cast<const unsigned long long*>(xs)[i];
#pragma unroll
        for (int j = 0; j < MC; ++j) {
          const unsigned long long yv = reinterpret_cast<const unsigned long long*>(ys)[j];
#pragma unroll
          for (int i = 0; i < MR; ++i) nt_fma2(p[i * MC + j], xv[i], yv);
        }
      }
      if (++folded == FOLD || nn == 0) {
        folded = 0;
#pragma unroll
        for (int i = 0; i < NQ; ++i) nt_fold2(acc[i], p[i]);
      }
      __syncwarp();
    }
    if (nn == 0) break;
    cn = nn;
    ckc = nkc;
    cxs = nxs;
    cys = nys;
    buf ^= 1;
  }
  // ---- combine the groups in order through the (now idle) stage buffers, write the tile ------
  __syncwarp();
  // sums in [group][NE], then their errors; two neighbouring entries at a time
  constexpr int NP = (NE + 1) & ~1;
  float* red = wbase + g * NP;
#pragma unroll
  for (int n = 0; n < NQ; ++n) {
    const int e = (mr * MR + n / MC) * tw + mc * MC + n % MC;
    if (mr * MR + n / MC < th && mc * MC + n % MC < tw) {
      red[e] = acc[n];
      red[S * NP + e] = __uint_as_float((unsigned int)p[n]);
    }
  }
  __syncwarp();
  float* cb = a.C + tile.coff;
  const int cnt = th * tw;
  const float rtw = 1.0f / (float)tw;
  for (int e = 2 * lane; e < cnt; e += 64) {
    float2 s = *reinterpret_cast<const float2*>(wbase + e), r = *reinterpret_cast<const float2*>(wbase + S * NP + e);
#pragma unroll
    for (int o = 1; o < S; ++o) {
      const float2 v = *reinterpret_cast<const float2*>(wbase + o * NP + e);
      const float2 u = *reinterpret_cast<const float2*>(wbase + (S + o) * NP + e);
      const float2 t = __fadd2_rn(s, v);
      const float2 bp = nt_sub2(t, s);
      r = __fadd2_rn(r, __fadd2_rn(__fadd2_rn(nt_sub2(s, nt_sub2(t, bp)), nt_sub2(v, bp)), u));
      s = t;
    }
    s = __fadd2_rn(s, r);
    const int i = __float2int_rz(((float)e + 0.5f) * rtw), j = e - i * tw;
    const bool wrap = j + 1 == tw;
    cb[(int64_t)i * tile.nj + j] = s.x;
    if (e + 1 < cnt) cb[(int64_t)(i + wrap) * tile.nj + (wrap ? 0 : j + 1)] = s.y;
  }
  __syncwarp();
}

// Micro-tile class of a tile edge: 0, 1 = 2 x (3, 5), 2 .. 4 = 4 x (3, 4, 5).
__device__ __forceinline__ int nt_class(int t) { return t <= 6 ? 0 : t <= 10 ? 1 : (t - 1) >> 2; }

// AHEAD: during a tile the warp already holds the next one's description and the number of the one
// after it, which hides both fetches.  With few tiles a warp in a heavy tile would hold two that idle
// warps could do, so below kNtAhead tiles a resident warp tiles are taken one at a time: space,
// 20-wide, N = 500 / 1100 / 2250 55 -> 43, 134 -> 114, 446 -> 409 us; from 12 tiles a warp on
// taking ahead is faster (plane, 10-wide, N = 2250 152 -> 145 us, N = 4000 294 -> 284 us).
template <bool AHEAD>
__global__ void __launch_bounds__(kNtWarps * 32, 4) mul_f32_nt_kernel(NtArgs a) {
  extern __shared__ __align__(128) float nsm[];  // [warp][buffer][kNtBuf]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* wbase = nsm + (size_t)w * 2 * kNtBuf;  // the warp's two stage buffers
  const uint32_t wsmem = (uint32_t)__cvta_generic_to_shared(wbase);
  wait_for_previous();
  unsigned int t = 0, tn = 0;
  NtTile nxt = {};
  if (AHEAD) {
    if (lane == 0) t = atomicAdd(a.counter, 1u);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t < a.ntiles) nxt = a.tiles[t];
    if (lane == 0) tn = atomicAdd(a.counter, 1u);
  }
  for (;;) {
    NtTile tile;
    if (AHEAD) {
      if (t >= a.ntiles) break;
      tile = nxt;
      t = __shfl_sync(0xffffffffu, tn, 0);
      if (t < a.ntiles) nxt = a.tiles[t];
      if (lane == 0) tn = atomicAdd(a.counter, 1u);
    } else {
      if (lane == 0) t = atomicAdd(a.counter, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t >= a.ntiles) break;
      tile = a.tiles[t];
    }
    const int rc = nt_class(tile.th), cc = nt_class(tile.tw);
#define SF_NT_CASE(R, GR, MR, Cc, GC, MC) \
  case R * 5 + Cc: nt_tile<GR, MR, GC, MC>(a, tile, wbase, wsmem, lane); break;
#define SF_NT_ROW(R, GR, MR)                                                                       \
  SF_NT_CASE(R, GR, MR, 0, 2, 3) SF_NT_CASE(R, GR, MR, 1, 2, 5) SF_NT_CASE(R, GR, MR, 2, 4, 3)      \
  SF_NT_CASE(R, GR, MR, 3, 4, 4) SF_NT_CASE(R, GR, MR, 4, 4, 5)
    switch (rc * 5 + cc) {
      SF_NT_ROW(0, 2, 3) SF_NT_ROW(1, 2, 5) SF_NT_ROW(2, 4, 3) SF_NT_ROW(3, 4, 4) SF_NT_ROW(4, 4, 5)
      default: break;
    }
#undef SF_NT_ROW
#undef SF_NT_CASE
  }
}

// One operand of the pre-pass: its blocks as stored and where the packed ones go.
struct NtPack {
  int64_t nb;
  const int32_t* bsize;
  const int32_t* brow;
  const int32_t* bcol;
  const int64_t* voff;
  const int64_t* poff;
  int trans;
  const float* src;
  float* dst;
};

// Blocks w0, w0 + nw, .. of an operand: block b (rows x cols, row-major in `src` at voff[b]), or its
// transpose (trans), is written at poff[b] as panels of at most 20 rows, [t / 2][row][t % 2] each,
// zeros for the padded t and up to the next multiple of 4 floats.  LANES lanes per block; a lane writes
// one pair of t (8 bytes) at a time.  A chain of dependent loads leads to each block: where there are
// many, kNtPackLanes lanes keep 4 blocks of a warp in flight (N = 50000 in the plane 183 us, a warp to
// a block 306).
constexpr int kNtPackLanes = 8;
template <int LANES>
__device__ __forceinline__ void nt_pack(const NtPack& p, int64_t w0, int64_t nw, int lane) {
  for (int64_t b = w0; b < p.nb; b += nw) {
    const int rows = p.bsize[p.brow[b]], cols = p.bsize[p.bcol[b]];
    const int R = p.trans ? cols : rows, K = p.trans ? rows : cols;  // panel rows and t extent
    const int rs = p.trans ? 1 : cols, ts = p.trans ? cols : 1;      // source strides of a row and of t
    const int kp = nt_even(K) >> 1;
    const float* __restrict__ s = p.src + p.voff[b];
    float2* __restrict__ d = reinterpret_cast<float2*>(p.dst + p.poff[b]);
    for (int r0 = 0; r0 < R; r0 += kTile) {
      const int th = min(kTile, R - r0);
      const float rth = 1.0f / (float)th;
#pragma unroll 4
      for (int e = lane; e < th * kp; e += LANES) {
        const int tp = e < (1 << 20) ? __float2int_rz(((float)e + 0.5f) * rth) : e / th, r = r0 + e - tp * th;
        const float* v = s + (int64_t)r * rs + (int64_t)(2 * tp) * ts;
        d[(int64_t)r0 * kp + e] = make_float2(v[0], 2 * tp + 1 < K ? v[ts] : 0.0f);
      }
    }
    if (lane == 0 && ((R * kp) & 1)) d[(int64_t)R * kp] = make_float2(0.0f, 0.0f);
  }
}

// Packed copies of both operands (y.nb = 0: one copy serves both sides), and zero in the product's
// tile counter.  Small products are bound by their launches, so the product's launch overlaps this
// one's (N = 1000 in the plane 83.2 -> 80.8 us), and where every block of an operand can have a
// warp at once it gets one, the second operand beside the first (grid row 1): 8 lanes a block took
// both operands in turn, 10 us each for 20-wide blocks (N = 500 in space, two operands 75 -> 53 us).
template <int LANES>
__global__ void nt_prepare_kernel(NtPack x, NtPack y, unsigned int* counter) {
  const int lane = threadIdx.x % LANES;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES;
  const int64_t nw = (int64_t)gridDim.x * blockDim.x / LANES;
  let_next_start();  // the product's CTAs take their places and wait
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *counter = 0u;
  if (blockIdx.y == 0) nt_pack<LANES>(x, w, nw, lane);
  if (blockIdx.y + 1 == gridDim.y) nt_pack<LANES>(y, w, nw, lane);
}

}  // namespace

// ---- host side --------------------------------------------------------------------------

// Float offsets of the packed blocks of pattern p (nblocks entries) on the device: rows x even t
// extent of the block or of its transpose, rounded up to 16 bytes.
static s_status padded_offsets(const s_pattern_t* p, bool trans, int64_t** out, int64_t* total) {
  const int64_t nb = p->d.nblocks;
  std::vector<int64_t> off(std::max<int64_t>(nb, 1), 0);
  int64_t s = 0;
  for (int64_t b = 0; b < nb; ++b) {
    off[b] = s;
    const int r = p->bsize[p->brow[b]], c = p->bsize[p->colidx[b]];
    s += ((int64_t)(trans ? c : r) * nt_even(trans ? r : c) + 3) & ~int64_t(3);
  }
  *total = s;
  SF_CUDA(cudaMalloc(out, sizeof(int64_t) * off.size()));
  SF_CUDA(cudaMemcpy(*out, off.data(), sizeof(int64_t) * off.size(), cudaMemcpyHostToDevice));
  return S_OK;
}

void nt_free_side(NtSideDesc* s) {
  cudaFree(s->poff);
  cudaFree(s->scratch);
  *s = NtSideDesc();
}

// Configure one side of the packed product: `pat` is the stored operand's pattern, `list` the
// row (X) or column (Y) lists of op(.), `trans` whether the packed slice is the transpose of
// the stored block.
static s_status nt_side(const s_pattern_t* pat, const Side& list, bool trans, NtSideDesc* s) {
  s->ptr = list.ptr;
  s->idx = list.idx;
  s->blk = list.blk;
  s->pat = pat;
  s->trans = trans;
  s_status st = padded_offsets(pat, trans, &s->poff, &s->len);
  if (st) return st;
  SF_CUDA(cudaMalloc(&s->scratch, sizeof(float) * std::max<int64_t>(s->len, 1)));
  s->off = s->poff;
  return S_OK;
}

static NtSide list_side(const NtSideDesc& s) { return NtSide{s.ptr, s.idx, s.blk, s.off}; }

void nt_free_lists(MulDesc* d) {
  cudaFree(d->nt_eptr);
  cudaFree(d->nt_ent);
  cudaFree(d->nt_tiles);
  d->nt_tiles = nullptr;
  d->nt_eptr = nullptr;
  d->nt_ent = nullptr;
  d->nt_ranges.clear();
}

// Counts the lists of a configured descriptor, lays out the ranges of blocks that go through the
// workspace together (one range: the plan keeps the lists, which are written here) and
// allocates.  All work is on the default stream and finished on return.
static s_status nt_build_lists(MulDesc* d) {
  for (auto kern : {mul_f32_nt_kernel<false>, mul_f32_nt_kernel<true>})
    SF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNtSmem));
  SF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&d->nt_per_sm, mul_f32_nt_kernel<true>, kNtWarps * 32, kNtSmem));
  d->nt_per_sm = std::max(d->nt_per_sm, 1);
  // the entries count operand offsets in 4 floats with 32 bits, t in 16
  if ((d->ntx.len >> 2) > (int64_t)UINT32_MAX || (d->nty.len >> 2) > (int64_t)UINT32_MAX) return S_OK;
  for (const s_pattern_t* q : {d->px, d->py})
    if (q->d.max_bsize > 65000) return S_OK;
  const s_pattern_t* C = d->pc;
  const int64_t nb = C->d.nblocks;
  // where each block's list and tiles start; on the device one buffer, whose second half holds the
  // lists' lengths first (allocations and copies are most of the time this takes for small plans)
  std::vector<int64_t> start(2 * (nb + 1), 0);
  int64_t *eptr = start.data(), *tptr = eptr + nb + 1;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((nb + 7) / 8, (int64_t)sm_count() * 64));
  SF_CUDA(cudaMalloc(&d->nt_eptr, sizeof(int64_t) * start.size()));
  if (nb > 0) {
    std::vector<int32_t> h(nb);
    int32_t* cnt = (int32_t*)(d->nt_eptr + nb + 1);
    nt_list_kernel<false><<<grid, 256>>>(list_side(d->ntx), list_side(d->nty), C->d.bsize, C->d.brow, C->d.colidx, 0, nb,
                                         cnt, nullptr, 0, nullptr);
    SF_CUDA(cudaGetLastError());
    SF_CUDA(cudaMemcpy(h.data(), cnt, sizeof(int32_t) * nb, cudaMemcpyDeviceToHost));
    for (int64_t k = 0; k < nb; ++k) {
      const int64_t ni = C->bsize[C->brow[k]], nj = C->bsize[C->colidx[k]];
      eptr[k + 1] = eptr[k] + h[k];
      tptr[k + 1] = tptr[k] + ((ni + kTile - 1) / kTile) * ((nj + kTile - 1) / kTile);
    }
  }
  SF_CUDA(cudaMemcpy(d->nt_eptr, start.data(), sizeof(int64_t) * start.size(), cudaMemcpyHostToDevice));
  SF_CUDA(cudaMalloc(&d->nt_tiles, sizeof(NtTile) * std::max<int64_t>(tptr[nb], 1)));
  if (nb > 0) {
    nt_tile_kernel<<<(unsigned)((nb + 255) / 256), 256>>>(nb, C->d.bsize, C->d.brow, C->d.colidx, C->d.voff,
                                                          d->nt_eptr + nb + 1, d->nt_eptr, d->nt_tiles);
    SF_CUDA(cudaGetLastError());
  }
  const int64_t total = eptr[nb], bytes = total * (int64_t)sizeof(NtEntry);
  size_t avail = 0, all = 0;
  if (bytes > kNtListLeast) SF_CUDA(cudaMemGetInfo(&avail, &all));
  const int64_t work = std::max(kNtListLeast, std::min(kNtListWork, (int64_t)(avail / 512))) / (int64_t)sizeof(NtEntry);
  int64_t most = bytes <= kNtListMax && (int64_t)avail - bytes >= (int64_t)(all / 2) ? total : work;  // entries of a range
  for (;; most = work) {
    int64_t room = 0;  // entries to allocate
    NtRange r{0, 0, 0, 0, 0};
    d->nt_ranges.clear();
    for (int64_t k = 0; k < nb; ++k) {
      // (a launch counts its tiles in 32 bits)
      if (r.k1 > r.k0 && (eptr[k + 1] - r.base > most || tptr[k + 1] - r.t0 > INT32_MAX)) {
        d->nt_ranges.push_back(r);
        r = NtRange{k, k, tptr[k], tptr[k], eptr[k]};
      }
      r.k1 = k + 1;
      r.t1 = tptr[k + 1];
      room = std::max(room, eptr[r.k1] - r.base);
    }
    if (nb > 0) d->nt_ranges.push_back(r);
    const cudaError_t e = cudaMalloc(&d->nt_ent, sizeof(NtEntry) * std::max<int64_t>(room, 1));
    if (e == cudaSuccess) break;
    d->nt_ent = nullptr;
    if (e != cudaErrorMemoryAllocation || most <= work) return cuda_error(e, "packed float product: lists");
    cudaGetLastError();  // room for all of them at once is not to be had: range by range
  }
  if (d->nt_ranges.size() == 1) {
    nt_list_kernel<true><<<grid, 256>>>(list_side(d->ntx), list_side(d->nty), C->d.bsize, C->d.brow, C->d.colidx, 0, nb,
                                        nullptr, d->nt_eptr, 0, d->nt_ent);
    SF_CUDA(cudaGetLastError());
  }
  SF_CUDA(cudaDeviceSynchronize());
  return S_OK;
}

// Packed sides of a float descriptor (forward or adjoint) for C = op(X) op(Y), op(X) = X^T
// when x_trans and op(Y) = Y^T when y_trans.  X side: op(X) rows; the stored
// block of a row-list entry is (nu, lambda) when op(X) = X (CSR row) and (lambda, nu) when
// op(X) = X^T (CSC column).  Y side: op(Y) columns; with op(Y) = Y^T the stored block of a
// CSR-row entry (nu', lambda) has a row per column of op(Y); with op(Y) = Y the CSC-column entry
// (lambda, nu') is transposed, unless `y_sym` (Y = X declared symmetric and called with one
// buffer) lets the kernel read Y(nu', lambda) through Y's own CSR rows.
static s_status nt_sides(MulDesc* d, bool x_trans, bool y_trans, bool y_sym) {
  const DevPattern& px = d->px->d;
  const DevPattern& py = d->py->d;
  Side xl = x_trans ? Side{px.colptr, px.rowidx, px.cscblk, px.voff, true}
                    : Side{px.rowptr, px.colidx, nullptr, px.voff, false};
  s_status st = nt_side(d->px, xl, x_trans, &d->ntx);
  if (st) return st;
  Side yl;
  bool ytrans;
  if (y_trans || y_sym) {
    yl = Side{py.rowptr, py.colidx, nullptr, py.voff, false};
    ytrans = false;
  } else {
    yl = Side{py.colptr, py.rowidx, py.cscblk, py.voff, true};
    ytrans = true;
  }
  if (!y_sym || x_trans) return nt_side(d->py, yl, ytrans, &d->nty);
  // B = A read through A's rows: the same packed blocks as the X side, one copy for both
  d->nty.ptr = yl.ptr;
  d->nty.idx = yl.idx;
  d->nty.blk = yl.blk;
  d->nty.pat = d->py;
  d->nty.off = d->ntx.off;
  d->nty.len = d->ntx.len;
  d->nty.from_x = true;
  return S_OK;
}

// Configures a descriptor for the packed kernel, or leaves it without packed copies and lists, all of
// them: the old ones go first, since lists say where blocks start in copies that are laid out
// anew.  Where device or host memory runs out the descriptor stays without them and the product
// runs on the tile kernel, which reads the operands as stored.
s_status nt_configure(MulDesc* d, bool x_trans, bool y_trans, bool y_sym) {
  nt_free_lists(d);
  nt_free_side(&d->ntx);
  nt_free_side(&d->nty);
  d->nt_ysym = y_sym;
  s_status st;
  try {
    st = nt_sides(d, x_trans, y_trans, y_sym);
    if (!st) st = nt_build_lists(d);
  } catch (const std::bad_alloc&) {
    st = S_ERR_NOMEM;
  }
  if (st || !d->nt_ent) {
    nt_free_lists(d);
    nt_free_side(&d->ntx);
    nt_free_side(&d->nty);
  }
  return st == S_ERR_NOMEM ? S_OK : st;
}

static NtPack pack_of(const NtSideDesc& s, const void* src) {
  const DevPattern& p = s.pat->d;
  return NtPack{p.nblocks, p.bsize, p.brow, p.colidx, p.voff, s.poff, s.trans ? 1 : 0, (const float*)src, s.scratch};
}

bool nt_usable(const MulDesc& d, const void* X, const void* Y) {
  if (!d.nt_ent || !d.ntx.off || !d.nty.off) return false;
  // a symmetric Y side reads B through A's rows: only valid for B = A
  return !d.nt_ysym || X == Y;
}

s_status launch_nt(const MulDesc& d, const void* X, const void* Y, void* C, cudaStream_t st) {
  if (d.ntiles == 0) return S_OK;
  s_status s = take_timeout(d);
  if (s) return s;
  const NtPack px = pack_of(d.ntx, X);
  const NtPack py = d.nty.from_x ? NtPack{} : pack_of(d.nty, Y);
  const int64_t nb = std::max(px.nb, py.nb), ctas = (int64_t)sm_count() * 16;  // 8 CTAs an SM are resident
  if (nb <= ctas * 8)
    nt_prepare_kernel<32><<<dim3((unsigned)std::max<int64_t>(1, (nb + 7) / 8), py.nb > 0 ? 2 : 1), 256, 0, st>>>(
        px, py, d.counter);
  else
    nt_prepare_kernel<kNtPackLanes><<<(unsigned)std::min((nb * kNtPackLanes + 255) / 256, ctas), 256, 0, st>>>(px, py,
                                                                                                             d.counter);
  const DevPattern& pc = d.pc->d;
  for (const NtRange& r : d.nt_ranges) {
    if (d.nt_ranges.size() > 1) {
      const int64_t lg = std::max<int64_t>(1, std::min<int64_t>((r.k1 - r.k0 + 7) / 8, (int64_t)sm_count() * 64));
      nt_list_kernel<true><<<(int)lg, 256, 0, st>>>(list_side(d.ntx), list_side(d.nty), pc.bsize, pc.brow, pc.colidx, r.k0,
                                                    r.k1, nullptr, d.nt_eptr, r.base, d.nt_ent);
    }
    NtArgs a;
    a.X = d.ntx.scratch;
    a.Y = d.nty.from_x ? d.ntx.scratch : d.nty.scratch;
    a.ent = d.nt_ent;
    a.base = r.base;
    a.tiles = d.nt_tiles + r.t0;
    a.ntiles = (uint32_t)(r.t1 - r.t0);
    a.counter = d.counter;
    a.C = (float*)C;
    if (r.k0 > 0) SF_CUDA(cudaMemsetAsync(d.counter, 0, sizeof(unsigned int), st));
    const int64_t want = (r.t1 - r.t0 + kNtWarps - 1) / kNtWarps;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * d.nt_per_sm);
    const bool ahead = r.t1 - r.t0 >= (int64_t)kNtAhead * sm_count() * d.nt_per_sm * kNtWarps;
    auto kern = ahead ? mul_f32_nt_kernel<true> : mul_f32_nt_kernel<false>;
    if (grid > 0) SF_CUDA(launch_overlapped(kern, dim3((unsigned)grid), kNtWarps * 32, kNtSmem, 0, st, a));
    SF_CUDA(cudaGetLastError());
  }
  return S_OK;
}

}  // namespace sf
