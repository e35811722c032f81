// Internal definitions shared by the translation units of libsformat.so.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "sformat.h"

namespace sf {

// Thread-local error message; set_error returns the status for `return set_error(...)`.
s_status set_error(s_status st, const std::string& msg);
s_status cuda_error(cudaError_t e, const char* what);
// SM count of the current device (cached per device ordinal).
int sm_count();

#define SF_CUDA(call)                                     \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return sf::cuda_error(e_, #call); \
  } while (0)

// Device copy of a block pattern (Sec. 3.3: cluster pairs of one tree), with the
// block-CSR rows and the transposed (block-CSC) index, both sorted.
struct DevPattern {
  int32_t nc = 0;
  int64_t n = 0;        // matrix dimension
  int64_t nblocks = 0;
  int64_t nnz = 0;
  int32_t max_bsize = 0;
  // device arrays
  int32_t* bsize = nullptr;   // nc
  int64_t* boff = nullptr;    // nc+1 row offsets
  int64_t* rowptr = nullptr;  // nc+1
  int32_t* colidx = nullptr;  // nblocks
  int32_t* brow = nullptr;    // nblocks: block row of each block
  int64_t* voff = nullptr;    // nblocks+1 entry offsets
  int64_t* colptr = nullptr;  // nc+1 (CSC)
  int32_t* rowidx = nullptr;  // nblocks: block rows of column, sorted
  int32_t* cscblk = nullptr;  // nblocks: CSR block index of each CSC entry
  int32_t* diag = nullptr;    // nc: block index of (nu,nu) or -1
  int32_t* roworder = nullptr;  // nc: block rows by falling number of blocks
  int32_t nlong = 0;            // the first nlong of them are long (kLongRow)
};

// Blocks of a row beyond which a cluster of CTAs shares it (add.cu); fewer where the matrix has at most
// two rows per SM, which would leave most of the GPU idle.
constexpr int kLongRow = 256, kLongRowSmall = 32;

}  // namespace sf

struct s_pattern_t {
  sf::DevPattern d;
  // host copies
  std::vector<int32_t> bsize, level, colidx, brow, diag;
  std::vector<int64_t> boff, rowptr, voff;
  uint64_t tree_hash = 0;
  bool has_all_diag = true;
};

namespace sf {

// One side of a masked product: op(X) with op = identity or transpose.  The index list
// of row nu of op(X) is idx[ptr[nu] .. ptr[nu+1]) with X block ids blk[...].
struct Side {
  const int64_t* ptr;
  const int32_t* idx;
  const int32_t* blk;  // nullptr: blk = position (CSR of X itself)
  const int64_t* voff;
  bool trans;
};

// Work item of the product kernels: one output tile of one block of C.
struct Tile {
  int32_t blk;  // C block id
  int16_t r0;   // first row of the tile inside the block
  int16_t c0;   // first column
};

// S_TF32X3 product (mul_tc.cu): MMA rows (member columns) and columns (own rows) of a panel,
// members per panel, lambda extent of one stage, widest block supported.
constexpr int kTcM = 128;
constexpr int kTcN = 32;
constexpr int kTcP = 8;
constexpr int kTcKC = 24;
constexpr int kTcMaxB = 96;

// One stage of an S_TF32X3 panel: source offsets (in the split value planes) of the X slice
// and of each member's Y slice (-1: member has no block for this lambda), lambda's block
// size (row pitch of the slices) and the staged extent.
struct TcEntry {
  int64_t x;
  int64_t y[kTcP];
  int32_t nl, wd;
};

// One operand side of the packed float product (mul_nt.cu): the op(X) row lists or op(Y)
// column lists, and the packed copy of the operand's blocks that a pre-pass of every product
// writes into `scratch` at offsets poff.
struct NtSideDesc {
  const int64_t* ptr = nullptr;
  const int32_t* idx = nullptr;
  const int32_t* blk = nullptr;
  const int64_t* off = nullptr;   // nullptr: side not configured
  const s_pattern_t* pat = nullptr;
  bool trans = false;             // the packed copy holds the stored blocks transposed
  bool from_x = false;            // Y side: reads the X side's packed copy (B = A, symmetric)
  int64_t* poff = nullptr;
  float* scratch = nullptr;
  int64_t len = 0;                // floats of the packed copy
};

// One matching lambda block (or piece of kNtKC values of t of a wide one) of a block of S_C in the
// packed float product: where the packed X and Y blocks start (in 4 floats), their padded t
// extent, the first t of the piece and its extent.
struct alignas(16) NtEntry {
  uint32_t xo, yo;
  uint16_t kp, t0;
  uint32_t kc;
};

// Output tile of the packed float product: where its list and its first entry of C start, list
// length, row pitch of C, place in the block and extent.
struct alignas(16) NtTile {
  int64_t e0, coff;
  int32_t ne, nj;
  uint16_t r0, c0, th, tw;
};

// Blocks k0 .. k1-1 of S_C (tiles t0 .. t1-1) whose lists are in memory together, from entry
// `base` on.
struct NtRange {
  int64_t k0, k1, t0, t1, base;
};

struct MulDesc {
  Side x, y;                 // C = op(X) op(Y) on S_C
  const s_pattern_t* pc;
  const s_pattern_t* px;
  const s_pattern_t* py;
  Tile* tiles = nullptr;     // device tile list, block order
  int64_t ntiles = 0;
  int edge = 20;             // tile edge of the list
  int variant = 0;           // float kernel variant (autotuned)
  Tile* ptiles = nullptr;    // row-panel variants: tiles ordered by (row, r0, column)
  int2* pidx = nullptr;      // per panel: first tile in ptiles, tile count
  int64_t npanels = 0;
  int panel_edge = 0, panel_size = 0;
  int64_t* tc_pstart = nullptr;  // S_TF32X3: first stage of each panel (npanels + 1)
  TcEntry* tc_ent = nullptr;     // S_TF32X3: stages of all panels
  int64_t tc_nentries = 0;
  float* tc_xh = nullptr;        // S_TF32X3 split planes (hi, lo) of both operands
  float* tc_xl = nullptr;
  float* tc_yh = nullptr;
  float* tc_yl = nullptr;
  unsigned int* err = nullptr;       // time-out word, device view: set to 1 when a bounded wait
  unsigned int* err_host = nullptr;  // of a kernel ran out; pinned host memory mapped into the
                                     // device, so the host reads it without a sync
  bool tc_sym = false;             // symmetric plan: B = A, Y read through its stored transpose
  NtSideDesc ntx, nty;             // packed float product sides (S_FP32)
  int64_t* nt_eptr = nullptr;      // first entry, then first tile, of each block of S_C (device, twice nblocks + 1)
  NtTile* nt_tiles = nullptr;      // tiles of S_C in block order
  NtEntry* nt_ent = nullptr;       // lists of the current range (nullptr: side or lists missing)
  std::vector<NtRange> nt_ranges;  // one: the plan keeps all lists
  int nt_per_sm = 1;               // resident CTAs of the packed kernel
  bool nt_ysym = false;            // Y side read through X's rows (B = A, symmetric)
  float2* df_x = nullptr;    // S_FP64_DF: split operands (hi, lo)
  float2* df_y = nullptr;
  struct __nv_bfloat16* bf_x = nullptr;  // S_BF16X3: three bfloat16 planes per operand
  struct __nv_bfloat16* bf_y = nullptr;
  unsigned int* counter = nullptr;  // device work counter
  int64_t triples = 0;
  double flops = 0.0;
};

s_status build_desc(const s_pattern_t* X, bool tx, const s_pattern_t* Y, bool ty, const s_pattern_t* C, s_prec prec,
                    MulDesc* d);
void free_desc(MulDesc* d);
s_status tc_prepare(MulDesc* d);
void tc_free(MulDesc* d);
s_status launch_tc(const MulDesc& d, const void* X, const void* Y, void* C, cudaStream_t st);
// S_ERR_TIMEOUT (and the record cleared) if the descriptor's time-out word is set, else S_OK.
s_status take_timeout(const MulDesc& d);
// Packed float product (mul_nt.cu): configure the sides and lists of a float descriptor, whether a call
// with these buffers can use it, the launch, and the release of its scratch.
s_status nt_configure(MulDesc* d, bool x_trans, bool y_trans, bool y_sym);
bool nt_usable(const MulDesc& d, const void* X, const void* Y);
s_status launch_nt(const MulDesc& d, const void* X, const void* Y, void* C, cudaStream_t st);
void nt_free_side(NtSideDesc* s);
void nt_free_lists(MulDesc* d);
s_status run_mul(const MulDesc& d, s_prec prec, const void* X, const void* Y, void* C, cudaStream_t st);

// Element-wise kernels (add.cu)
s_status run_add(const s_pattern_t* p, s_prec prec, double alpha, const void* A, double beta, const void* B,
                 double gamma, void* C, cudaStream_t st);
// Y = A X for nvec vectors (N x nvec, column-major)
s_status run_spmm_f64(const s_pattern_t* p, const double* A, const double* X, int nvec, double* Y, cudaStream_t st);
// `iters` power steps on x (all ones at first) and y, N doubles each; sc: kPowerWork doubles,
// sc[0] = the last Rayleigh quotient
constexpr int kRedCtas = 256;                 // partial sums of a reduction
constexpr int kPowerWork = 2 + 2 * kRedCtas;
s_status run_power(const s_pattern_t* p, const double* A, int iters, double* x, double* y, double* sc, cudaStream_t st);
// part[0 .. kRedCtas) = partial sums of a b, part[kRedCtas .. 2 kRedCtas) of b b (fixed order; the
// caller adds them in order)
s_status run_dot2(int64_t n, const double* a, const double* b, double* part, cudaStream_t st);
// the partial sums of a plain sum of a, as the first half of run_dot2's
s_status run_sum(int64_t n, const double* a, double* part, cudaStream_t st);

constexpr int kTile = 20;  // output tile edge of the product kernels

// Asynchronous copies global -> shared of 8 and 16 bytes.
__device__ __forceinline__ void d64_cp(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void d64_cp2(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// rows x cols doubles at row pitch ld -> dst, packed; one warp.  A packed source on 16-byte
// boundaries goes two doubles to a copy.
__device__ __forceinline__ void d64_stage(uint32_t dst, const double* src, int rows, int cols, int ld, int lane) {
  const int len = rows * cols;
  if (cols == ld) {
    if (((dst | (uint32_t)reinterpret_cast<uintptr_t>(src)) & 15) == 0) {
      for (int e = 2 * lane; e + 1 < len; e += 64) d64_cp2(dst + 8u * (uint32_t)e, src + e);
      if ((len & 1) && lane == 0) d64_cp(dst + 8u * (uint32_t)(len - 1), src + len - 1);
    } else {
#pragma unroll 4
      for (int e = lane; e < len; e += 32) d64_cp(dst + 8u * (uint32_t)e, src + e);
    }
  } else {
    const float rc = 1.0f / (float)cols;
    for (int e = lane; e < len; e += 32) {
      const int r = __float2int_rz(((float)e + 0.5f) * rc);
      d64_cp(dst + 8u * (uint32_t)e, src + (int64_t)r * ld + (e - r * cols));
    }
  }
}

// Programmatic dependent launch, for chains of short kernels (a dependent launch costs about 2 us
// between the kernels, and each kernel starts with a chain of loads of plan data).  A kernel
// launched by launch_overlapped may start once every CTA of the stream's previous kernel has called
// let_next_start() or left; it may read plan data at once, but must call wait_for_previous() (in
// thread blocks that do work, and in at least one) before it reads or writes anything an earlier
// kernel of the stream touches.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// `cluster` CTAs to a cluster (0: none).
template <class... Par, class... Arg>
cudaError_t launch_overlapped(void (*kern)(Par...), dim3 grid, int threads, size_t smem, unsigned cluster,
                              cudaStream_t st, Arg... args) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<Par>(args)...);
}

}  // namespace sf

struct s_plan_t {
  s_prec prec;
  const s_pattern_t* a;
  const s_pattern_t* b;
  const s_pattern_t* c;
  sf::MulDesc fwd;
  sf::MulDesc adjA;  // dA = P_{S_A}(dC B^T), built on first use
  sf::MulDesc adjB;  // dB = P_{S_B}(A^T dC)
  bool adj_built = false;
  float tune_ms[16] = {0};
};
