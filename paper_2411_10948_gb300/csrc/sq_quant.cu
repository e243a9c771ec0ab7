// ShiftQuant quantizer kernels for sm_103a and their C entry points.
//
//   range pass  (Sec. 3.1)   per-column max|x| with 128-bit loads and an atomic max on the
//                            bit pattern of the non-negative float; per-row max for the
//                            per-in-channel weight role
//   grouping    (Eq. 3)      tau_0 = max_c r_c, e_c = the largest e <= N_G-1 with
//                            r_c 2^e <= tau_0, i.e. floor(log2(tau_0 / r_c)) clipped
//   quantize    (App. D/B)   q = round(x 2^e_c Q / tau_0) with round-to-nearest-even or
//                            stochastic rounding on a counter-based SplitMix64 draw;
//                            optional shift of weight codes by 2^(N_G-1-e) (ShiftMM)
//
// All three are HBM-bound streaming passes.  The quantizer writes the codes directly in
// the operand format of the tensor-core GEMM (E4M3 or BF16, exact integers) and, in the
// same pass, the transposed copy the weight-gradient GEMM reads, staged through shared
// memory so both writes stay coalesced.
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>

#include "sq_device.cuh"
#include "sq_host.h"
#include "sq_quant_dev.cuh"

namespace sq {

static thread_local char g_last_error[512];

int fail(int status, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_last_error, sizeof g_last_error, fmt, ap);
  va_end(ap);
  return status;
}

static void clear_error() { g_last_error[0] = 0; }

// the group order a shiftquant_quantize_ordered call hands to the quantizer launch it makes
// (per host thread; null outside such a call)
static thread_local const int* g_order_cols = nullptr;
static thread_local const int* g_order_rows = nullptr;

// ===================================================================== range pass
constexpr int kColTx = 32;  // threads along columns, 4 columns each: 128 columns per block
constexpr int kColTy = 8;   // threads along rows

__device__ __forceinline__ uint32_t abs_bits(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }

// range_bits[c] = max over this block's rows of |x[r, c]| as an ordered bit pattern
// (for non-negative floats, larger value <=> larger unsigned pattern; NaN sorts above Inf).
// zero the range accumulators a[na] and b[nb] (b may be null); the range pass that follows
// may launch at once: it reads x first and these only after its wait
__global__ void __launch_bounds__(256)
    calib_init_kernel(unsigned* __restrict__ a, int64_t na, unsigned* __restrict__ b, int64_t nb) {
  griddep_launch_dependents();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < na; i += stride)
    a[i] = 0u;
  if (b != nullptr)
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nb; i += stride)
      b[i] = 0u;
}

// Grouping (Eq. 3) by one block of THREADS threads from the per-channel range bits:
// tau_0 = the largest range, then every channel's exponent; tau0_out receives tau_0 and
// the status word the non-finite flag.  Thread t holds channels t, t + THREADS, ... (up to
// kGroupPerThread of them in registers, so all its loads are in flight together; wider
// tensors read the rest twice).  Small blocks start faster, large ones take wide tensors
// in one round of loads.  Launched behind the range pass with programmatic stream
// serialization, it waits for the range pass before reading anything.
constexpr int kGroupPerThread = 16;
constexpr int kGroupSmallThreads = 256;
constexpr int kGroupLargeThreads = 1024;

template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    group_kernel(const unsigned* range_bits, int64_t C, int G,
                 float* __restrict__ tau0_out, uint8_t* __restrict__ exp_out,
                 int* __restrict__ status) {
  __shared__ unsigned wmax[THREADS / 32];
  __shared__ unsigned tau_bits;
  griddep_wait();
  griddep_launch_dependents();
  const int tid = threadIdx.x;
  unsigned v[kGroupPerThread];
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < kGroupPerThread; ++k) {
    const int64_t c = tid + static_cast<int64_t>(k) * THREADS;
    v[k] = c < C ? __ldcg(range_bits + c) : 0u;
    m = max(m, v[k]);
  }
  constexpr int64_t kHeld = static_cast<int64_t>(THREADS) * kGroupPerThread;
  for (int64_t c = kHeld + tid; c < C; c += THREADS) m = max(m, __ldcg(range_bits + c));
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((tid & 31) == 0) wmax[tid >> 5] = m;
  __syncthreads();
  if (tid < 32) {
    const unsigned w = __reduce_max_sync(0xFFFFFFFFu, tid < THREADS / 32 ? wmax[tid] : 0u);
    if (tid == 0) tau_bits = w;
  }
  __syncthreads();
  const unsigned tb = tau_bits;
  const float tau = __uint_as_float(tb);
  const bool nonfinite = tb >= 0x7F800000u;
#pragma unroll
  for (int k = 0; k < kGroupPerThread; ++k) {
    const int64_t c = tid + static_cast<int64_t>(k) * THREADS;
    if (c < C) exp_out[c] = static_cast<uint8_t>(nonfinite ? 0 : group_exponent(__uint_as_float(v[k]), tau, G));
  }
  for (int64_t c = kHeld + tid; c < C; c += THREADS)
    exp_out[c] = static_cast<uint8_t>(nonfinite ? 0 : group_exponent(__uint_as_float(__ldcg(range_bits + c)), tau, G));
  if (tid == 0) {
    *tau0_out = tau;
    if (nonfinite) atomicOr(status, kDevNonFinite);
  }
}

// A tensor as the range pass reads it.  A dense tensor whose rows are not 16-byte aligned is
// folded: `fold` rows (2 or 4, so that they make whole 16-byte vectors) become one row of
// fold x cols columns, whose column c stands for column c mod creal, plus `tail` elements of a
// last partial row; every load is then an aligned vector.  Other unaligned tensors are read
// element by element, the lanes on consecutive columns.
enum ViewForm { kViewVec, kViewFolded, kViewStrided };

struct RangeView {
  const float* x;
  int64_t R, C, ld;
  int form;        // ViewForm
  int64_t creal;   // columns of the tensor (C / creal rows are folded into one)
  int64_t tail;    // elements of the partial row R (folded tensors)
};

// The column maxima (ordered bit patterns of |x|: for non-negative floats a larger value is a
// larger pattern, NaN above Inf) of the thread's part of one tile of tc = 4 << lg columns by 8
// passes of 1024 / tc rows from r0 on: four columns -- quad qc, or in strided views columns
// qc + k 2^lg -- of rows r0 + u rpp, with all eight 16-byte loads in flight together.
// ROWS: rm[u] becomes the maximum with row u's four values.
// (x is complete before the kernel ahead of a range pass lets it launch, so single elements may
// come through the read-only path.)
template <bool ROWS, int FORM>
__device__ __forceinline__ void tile_maxima(const RangeView& t, int lg, int64_t cb, int64_t r0, int qc,
                                            unsigned (&m)[4], unsigned (&rm)[8]) {
  const int rpp = (kColTx * kColTy) >> lg;
  const int64_t c0 = cb + 4 * qc;
  if (FORM != kViewStrided && c0 + 3 < t.C) {
    // rows past the end re-read the last row, which leaves a maximum unchanged
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = ld_stream_v4(t.x + min(r0 + u * rpp, t.R - 1) * t.ld + c0);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned a[4] = {abs_bits(v[u].x), abs_bits(v[u].y), abs_bits(v[u].z), abs_bits(v[u].w)};
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = max(m[k], a[k]);
      if (ROWS) rm[u] = max(rm[u], max(max(a[0], a[1]), max(a[2], a[3])));
    }
    if (FORM == kViewFolded && t.tail > 0 && r0 + 8 * rpp > t.R) {   // the last row tile takes the partial row too
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (c0 + k < t.tail) m[k] = max(m[k], abs_bits(__ldg(t.x + t.R * t.ld + c0 + k)));
    }
    return;
  }
  if (FORM == kViewFolded) return;   // whole quads only
  const int64_t first = FORM == kViewVec ? c0 : cb + qc;   // (kViewVec: the last columns of padded rows)
  const int step = FORM == kViewVec ? 1 : 1 << lg;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const float* row = t.x + min(r0 + u * rpp, t.R - 1) * t.ld;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t c = first + k * step;
      const unsigned a = c < t.C ? abs_bits(__ldg(row + c)) : 0u;
      m[k] = max(m[k], a);
      if (ROWS) rm[u] = max(rm[u], a);
    }
  }
}

// the thread's column maxima to red[row pass ro][column]
template <int FORM>
__device__ __forceinline__ void put_maxima(unsigned* red, int lg, int ro, int qc, const unsigned (&m)[4]) {
  const int tc = 4 << lg;
#pragma unroll
  for (int k = 0; k < 4; ++k) red[ro * tc + (FORM != kViewStrided ? 4 * qc + k : qc + (k << lg))] = m[k];
}

// the accumulator of view column c
template <int FORM>
__device__ __forceinline__ unsigned* column_bits(unsigned* bits, const RangeView& t, int64_t c) {
  return bits + (FORM == kViewFolded ? c % t.creal : c);
}

// the maximum of tile column `col` over the block's row passes
__device__ __forceinline__ unsigned get_maximum(const unsigned* red, int lg, int col) {
  const int tc = 4 << lg, rpp = (kColTx * kColTy) >> lg;
  unsigned m = 0;
  for (int y = 0; y < rpp; ++y) m = max(m, red[y * tc + col]);
  return m;
}

// Range pass: block (x, y) reads tile (y, x) of TC = 4 << lg columns (the column count
// rounded up to a power of two, 4 to 128) by 8 passes of 1024 / TC rows, and sends its
// per-column maxima to range_bits with one atomic max per column.  Same-address atomics from
// hundreds of tiles of a narrow tensor serialise in L2, so narrow tensors (CL =
// kRangeCluster) run in clusters of CL blocks along the rows: each block merges its maxima
// into the first block of its cluster with atomic maxima on that block's shared memory, and
// only that block sends them on.  Wide tensors (CL = 1) spread their atomics over many
// addresses and run without clusters, which schedule more slowly.  Grids taller than the
// 65535-block limit walk the extra tiles in steps of gridDim.y.
// ROWS: the range pass of a weight for both of its roles -- also every row's max|x| over
// all columns (the per-in-channel ranges), each warp's eight rows of a tile reduced across
// its lanes and sent to row_bits with one atomic max per row and column block.
constexpr int kRangeCluster = 8;
constexpr int64_t kRangeClusterMaxCols = 512;   // clusters for tensors of at most 512 columns

template <int CL, bool ROWS, int FORM>
__global__ void __launch_bounds__(kColTx* kColTy)
    colmax_kernel(const RangeView v, int lg, unsigned* __restrict__ range_bits,
                  unsigned* __restrict__ row_bits, int* __restrict__ status) {
  __shared__ unsigned red[kColTy * kColTx * 4];
  __shared__ unsigned cmax[CL > 1 ? kColTx * 4 : 1];   // the cluster's maxima (first block)
  const int tid = threadIdx.y * kColTx + threadIdx.x;
  const int tc = 4 << lg, rpp = (kColTx * kColTy) >> lg;
  const int qc = tid & ((1 << lg) - 1), ro = tid >> lg;
  const int64_t cb = static_cast<int64_t>(blockIdx.x) * tc;
  const int64_t tile_rows = 8 * static_cast<int64_t>(rpp);
  const int64_t tiles = (v.R + tile_rows - 1) / tile_rows;
  if (CL > 1) {
    if (tid < kColTx * 4) cmax[tid] = 0u;
    cluster_arrive_release();   // the zeroed cmax is visible to the cluster after the wait
  }
  unsigned m[4] = {0u, 0u, 0u, 0u};
  bool row_bad = false;
#pragma unroll 1
  for (int64_t t = blockIdx.y; t < tiles; t += gridDim.y) {
    const int64_t r0 = t * tile_rows + ro;   // this thread's rows: r0 + u rpp
    unsigned rm[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};   // ROWS: this thread's columns of each of its rows
    tile_maxima<ROWS, FORM>(v, lg, cb, r0, qc, m, rm);
    if (ROWS) {
      // (lg = 5: a warp's 32 quads are one row of the tile, a warp row per pass)
      // the row accumulators are zeroed by the preceding kernel, which must have completed
      griddep_wait();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned w = __reduce_max_sync(0xFFFFFFFFu, rm[u]);
        const int64_t r = r0 + u * rpp;
        if (threadIdx.x == 0 && r < v.R && w != 0u) {
          atomicMax(row_bits + r, w);
          row_bad |= w >= 0x7F800000u;
        }
      }
    }
  }
  if (ROWS && row_bad) atomicOr(status, kDevNonFinite);
  // x has been read: the next kernel (the grouping) may start launching
  griddep_launch_dependents();
  put_maxima<FORM>(red, lg, ro, qc, m);
  __syncthreads();
  // thread t < tc: column t of the tile
  unsigned w = tid < tc ? get_maximum(red, lg, tid) : 0u;
  if (CL > 1) {
    cluster_wait_acquire();
    if (tid < tc && w != 0) red_max_cluster_u32(mapa_shared(smem_u32(cmax), 0) + tid * 4, w);
    cluster_arrive_release();
    cluster_wait_acquire();   // every block's maxima are in the first block's cmax
    if (cluster_ctarank() != 0) return;
    if (tid < tc) w = cmax[tid];
  }
  if (tid >= tc) return;
  // the accumulators are zeroed by the preceding kernel, which must have completed
  griddep_wait();
  const int64_t c = cb + tid;
  if (c < v.C && w != 0) {
    atomicMax(column_bits<FORM>(range_bits, v, c), w);
    if (w >= 0x7F800000u) atomicOr(status, kDevNonFinite);
  }
}

// The range pass of a wide weight (more than 512 columns) for both roles: per-column and
// per-row max|x|.  A block takes one tile of 64 rows (8 passes of 8) and walks kWeightRun
// consecutive 128-column blocks of it, one after another: each column block's maxima leave
// by atomics as in colmax_kernel, but every row's maximum leaves the block once per run.
// A block per column block would send each row cblocks atomics, and the blocks of one row
// tile send them together: on [4096, 11008] those 86 same-address atomics per row queued
// in L2 and took the pass from 33 us (columns alone) to 55 us; with runs of 4 it takes
// 36.5 us (measured, a scratch probe; prefetching the next column block into registers was
// slower).
constexpr int kWeightRun = 4;

// one row tile's run of column blocks j0 .. j0 + run - 1; *bad: a non-finite value was met
template <int FORM>
__device__ __forceinline__ void weight_range_run(const RangeView& v, int64_t tile, int64_t j0, int run, unsigned* red,
                                                 unsigned* __restrict__ col_bits,
                                                 unsigned* __restrict__ row_bits, bool* bad) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x, tx = tid & 31, ty = tid >> 5;
  const int64_t cblocks = (v.C + 4 * kColTx - 1) / (4 * kColTx);
  const int64_t r0 = tile * 8 * kColTy + ty;   // this thread's rows: r0 + u kColTy
  unsigned rm[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll 1
  for (int64_t j = j0; j < j0 + run && j < cblocks; ++j) {
    unsigned m[4] = {0u, 0u, 0u, 0u};
    const int64_t cb = j * 4 * kColTx;
    tile_maxima<true, FORM>(v, 5, cb, r0, tx, m, rm);
    put_maxima<FORM>(red, 5, ty, tx, m);
    __syncthreads();
    griddep_wait();   // the accumulators are zeroed by the preceding kernel
    if (tid < 4 * kColTx) {
      const unsigned w = get_maximum(red, 5, tid);
      const int64_t c = cb + tid;
      if (c < v.C && w != 0u) {
        atomicMax(col_bits + c, w);
        *bad |= w >= 0x7F800000u;
      }
    }
    __syncthreads();  // red is rewritten by the next column block
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const unsigned w = __reduce_max_sync(0xFFFFFFFFu, rm[u]);
    const int64_t r = r0 + u * kColTy;
    if (tx == 0 && r < v.R && w != 0u) {
      atomicMax(row_bits + r, w);
      *bad |= w >= 0x7F800000u;
    }
  }
}

template <int FORM>
__global__ void __launch_bounds__(kColTx* kColTy, 4)
    weight_range_kernel(const RangeView v, unsigned* __restrict__ col_bits, unsigned* __restrict__ row_bits,
                        int* __restrict__ status) {
  __shared__ unsigned red[kColTy * kColTx * 4];
  const int64_t tiles = (v.R + 8 * kColTy - 1) / (8 * kColTy);
  bool bad = false;
#pragma unroll 1
  for (int64_t t = blockIdx.y; t < tiles; t += gridDim.y)
    weight_range_run<FORM>(v, t, static_cast<int64_t>(blockIdx.x) * kWeightRun, kWeightRun, red, col_bits, row_bits, &bad);
  // x has been read: the next kernel may start launching
  griddep_launch_dependents();
  if (bad) atomicOr(status, kDevNonFinite);
}

// one warp per row: range[r] = max_c |x[r, c]|
__global__ void __launch_bounds__(256)
    rowmax_kernel(const float* __restrict__ x, int64_t R, int64_t C, int64_t ld, int vec,
                  float* __restrict__ range, int* __restrict__ status) {
  const int lane = threadIdx.x & 31;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (r >= R) return;
  const float* row = x + r * ld;
  unsigned m = 0;
  int64_t c = 0;
  if (vec) {
    const int64_t c4 = C & ~int64_t(3);
#pragma unroll 4
    for (int64_t cc = lane * 4; cc < c4; cc += 128) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(row + cc));
      m = max(max(m, abs_bits(v.x)), max(abs_bits(v.y), max(abs_bits(v.z), abs_bits(v.w))));
    }
    c = c4;
  }
  for (int64_t cc = c + lane; cc < C; cc += 32) m = max(m, abs_bits(__ldg(row + cc)));
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if (lane == 0) {
    range[r] = __uint_as_float(m);
    if (m >= 0x7F800000u) atomicOr(status, kDevNonFinite);
  }
}

// ======================================================================= quantize
// tau_0 of a tensor whose range pass ran in a layer's launch: the blocks send their maxima to
// kTauSlots words in turn (one word would take thousands of same-address atomics), and a
// reader takes the largest
constexpr int kTauSlots = 16;

__device__ __forceinline__ unsigned slots_word(const unsigned* slots) {   // the lane's word, of a whole warp
  const int lane = threadIdx.x & 31;
  return __ldcg(slots + (lane < kTauSlots ? lane : 0));
}
__device__ __forceinline__ float slots_tau(unsigned word) { return __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, word)); }

struct QuantArgs {
  const float* x;
  int64_t R, C, ld;
  int Q, G;
  uint64_t seed;
  int64_t row0;           // the tensor's first row within the logical tensor (SR index)
  const float* rt;        // &tau_0 (SHIFT) or range[] (PER_COL / PER_ROW)
  const unsigned* tslots; // SHIFT: tau_0 as the maximum of kTauSlots bit patterns (or null: *rt) ...
  float* tau_out;         // ... and stored here
  const uint8_t* exp;     // SHIFT: e_c, or null: formed from crange and tau_0
  const float* crange;    // ... the channel ranges
  uint8_t* exp_out;       // ... and written here by the first tile row
  const uint8_t* fold;    // exponents of the other GEMM operand, or null: formed from
  const float* frange;    // ... its channel ranges
  const unsigned* ftslots;   // ... and tau_0 (kTauSlots bit patterns)
  void* codes;
  int64_t ldc;
  void* codes_t;
  int64_t ldt;
  float* scale_out;
  int vec_in;             // 16-byte aligned input rows ...
  int sectors;            // ... that start on a sector
  int vec_out, vec_t;      // output rows that take four codes, or 16 transposed bytes, in one store
  int lg;                 // tiles of 4 << lg columns by 64 << (5 - lg) rows
  int form, fast;         // Form, and whether the tensor has what its register path needs
  // The launch runs beside the quantizer launch before it (a layer's tensors): that one let it
  // launch only after its own wait, so what both read is complete; the wait comes last, and
  // whoever waits for this launch has then waited for that one too.
  int beside;
  // group order of the GEMM inner index (or null): codes column c goes to pos_cols[c]
  // (ShiftQuant and per-row grans), codes_t column r to pos_rows[r] (per-column gran)
  const int* pos_cols;
  const int* pos_rows;
};

// Quantize tile: 8192 elements by 256 threads, tc = 4 << lg columns (128, 64 or 32) by
// 64 << (5 - lg) rows.  The rows form chunks of 8; a thread owns four consecutive columns of
// one chunk (a warp: 32 >> lg chunks).  Two ways through a tile:
//   registers: a tile inside the tensor whose rows are aligned (or shifted into place, or
//     whose codes go to a group order: Form), the thread's eight loads in flight together,
//     its rows unrolled.  Straight-line code that every thread runs once is bound by
//     instruction fetch as soon as tests are spread through it (with the edges handled in the
//     unrolled body: 8.4 cycles of no-instruction stall per issue, [12544, 256] 12.4 us against
//     8.7), so this path holds nothing but the common case;
//   shared memory: everything else.  Each warp copies its rows asynchronously -- 16 bytes a
//     copy where they are aligned, else one float a copy, the lanes on consecutive columns,
//     zeros outside the tensor -- and walks them in a rolled loop.
// Narrower tiles than 128 columns serve tensors whose column count would leave a 128-column
// grid partly idle (tile_lg).
constexpr int kQuantThreads = 256;
constexpr int kTileElems = 8192;
constexpr int kWarpBytes = kTileElems / 8 * 4;   // a warp's part of the tile in shared memory

static int64_t tile_cols(int lg) { return int64_t(4) << lg; }
static int64_t tile_rows(int lg) { return int64_t(64) << (5 - lg); }

// The widest tile (128, 64 or 32 columns) whose padded column count is within 1/8 of the
// best: the quantizer reads 512, 256 or 128 contiguous bytes a row, so wide tiles win unless
// they idle (147 columns: 256, 192, 160 padded).
static int tile_lg(int64_t C) {
  int64_t pad[3], best = INT64_MAX;
  for (int k = 0; k < 3; ++k) {
    const int64_t tc = tile_cols(5 - k);
    pad[k] = (C + tc - 1) / tc * tc;
    if (pad[k] < best) best = pad[k];
  }
  for (int k = 0; k < 2; ++k)
    if (pad[k] <= best + best / 8) return 5 - k;
  return 3;
}

// n codes as 32-bit words, the first code in the low bits
template <typename CodeT, int N>
__device__ __forceinline__ void encode_words(const float (&q)[N], uint32_t (&w)[N * sizeof(CodeT) / 4]) {
  if constexpr (sizeof(CodeT) == 2) {
#pragma unroll
    for (int k = 0; k < N / 2; ++k)
      w[k] = __byte_perm(__float_as_uint(q[2 * k]), __float_as_uint(q[2 * k + 1]), 0x7632);
  } else {
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
      const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(q[4 * k], q[4 * k + 1]), __NV_SATFINITE, __NV_E4M3);
      const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(q[4 * k + 2], q[4 * k + 3]), __NV_SATFINITE, __NV_E4M3);
      w[k] = lo | (hi << 16);
    }
  }
}

// Round to nearest even; + 0 turns a negative zero into a zero code.  |x| <= range gives
// |v| <= Q (1 + 2^-23), so rint never leaves [-Q, Q].
__device__ __forceinline__ float round_nearest(float v) { return __fadd_rn(rintf(v), 0.0f); }

// Stochastic rounding on the draw of generator state z, clamped to [-Q, Q].  The sum
// v + 1.5 2^23 rounded down has spacing 1, so l is floor(v) exactly for |v| < 2^22 (and +0
// for a zero); beyond, l stays on v's side of [-Q, Q] and the clamp decides.
__device__ __forceinline__ float round_stochastic(float v, uint64_t z, float Qf) {
  const float l = __fadd_rn(__fadd_rd(v, 12582912.0f), -12582912.0f);
  const float frac = __fsub_rn(v, l);
  const float u = __fmul_rn(static_cast<float>(splitmix64_top24(z)), 5.9604644775390625e-08f);  // * 2^-24, exact
  const float q = u < frac ? __fadd_rn(l, 1.0f) : l;
  return fminf(fmaxf(q, -Qf), Qf);
}

// the exponent of channel c: given, or formed from its range and tau_0
__device__ __forceinline__ int channel_exponent(float r, float tau, int G) {
  return isfinite(tau) ? group_exponent(r, tau, G) : 0;
}

// Q / range of a per-channel scale; 0 and *zero for a channel that quantizes to zero
__device__ __forceinline__ float channel_inv(float rg, float Qf, bool* zero) {
  const float inv = __fdiv_rn(Qf, rg);
  *zero = !(rg > 0.0f) || !isfinite(rg) || !isfinite(inv);
  return *zero ? 0.0f : inv;
}

// What gives the exponent of channel i: itself where it is given, else the channel's range
__device__ __forceinline__ uint32_t load_exponent(const uint8_t* exp, const float* range, int64_t i) {
  return exp != nullptr ? static_cast<uint32_t>(ld_here(exp + i)) : __float_as_uint(__ldcg(range + i));
}
__device__ __forceinline__ int exponent_of(uint32_t v, const uint8_t* exp, float tau, int G) {
  return exp != nullptr ? static_cast<int>(v) : channel_exponent(__uint_as_float(v), tau, G);
}

// Four columns' values from p: one load where they are all there (whole) and aligned, else those
// at the offsets at.  Past L1 a load of one column in four fetches the other three's sectors too:
// transposed codes of a [3072, 768] weight (4-bit) 4.7 us with four loads, 3.5 us with one.
__device__ __forceinline__ void load_ranges(const float* p, bool whole, const int (&at)[4], float (&v)[4]) {
  if (whole && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    const float4 f = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = f.x;
    v[1] = f.y;
    v[2] = f.z;
    v[3] = f.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = __ldcg(p + at[j]);
  }
}
__device__ __forceinline__ void load_exponents(const uint8_t* exp, const float* range, int64_t c0, bool whole,
                                               const int (&at)[4], uint32_t (&v)[4]) {
  if (exp == nullptr) {
    float f[4];
    load_ranges(range + c0, whole, at, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = __float_as_uint(f[j]);
  } else if (whole && (reinterpret_cast<uintptr_t>(exp + c0) & 3) == 0) {
    const uint32_t w = static_cast<uint32_t>(ld_here(reinterpret_cast<const int*>(exp + c0)));
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (w >> (8 * j)) & 0xFFu;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = static_cast<uint32_t>(ld_here(exp + c0 + at[j]));
  }
}

// The per-row values of a chunk's eight rows, held one row per lane of each group of eight
// lanes and handed round by shuffles: the multiplier (PER_ROW: Q / range) and the folded
// shift (PER_COL).
struct RowValues {
  float mul, fold;
  unsigned zero;  // bit i: row i of the lane's group quantizes to zero
};

// The thread's place in the tile at (bx, by).
struct TilePos {
  int chunk, col;   // its chunk, and its first column in the tile
  int64_t r, c;     // its first row and column in the tensor
};

__device__ __forceinline__ TilePos tile_pos(int lg, unsigned bx, unsigned by) {
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  TilePos p;
  p.chunk = (wq << (5 - lg)) + (lane >> lg);
  p.col = 4 * (lane & ((1 << lg) - 1));
  p.r = (static_cast<int64_t>(by) << (11 - lg)) + p.chunk * 8;
  p.c = (static_cast<int64_t>(bx) << (lg + 2)) + p.col;
  return p;
}

// This warp's rows of x into its part of the tile: the thread's quad of row i of its chunk
// ends up at its slot i (quad_slot).
__device__ __forceinline__ uint32_t quad_slot(uint32_t warp_smem, int lg, int i) {
  const int lane = threadIdx.x & 31;
  // row (lane >> lg) 8 + i of the warp's rows, quad (lane mod 2^lg) of the row
  return warp_smem + ((((lane >> lg) * 8 + i) << lg) + (lane & ((1 << lg) - 1))) * 16;
}

__device__ __forceinline__ void load_tile(const QuantArgs& a, unsigned bx, unsigned by, uint32_t warp_smem) {
  const int lg = a.lg;
  const TilePos p = tile_pos(lg, bx, by);
  if (a.vec_in && (static_cast<int64_t>(bx) + 1) << (lg + 2) <= a.C) {
    const float* src = a.x + p.r * a.ld + p.c;
    const uint32_t dst = quad_slot(warp_smem, lg, 0), step = 16u << lg;
    if (p.r + 8 <= a.R) {
#pragma unroll
      for (int i = 0; i < 8; ++i) cp_async_16(dst + i * step, src + i * a.ld, true);
    } else {
#pragma unroll 1
      for (int i = 0; i < 8; ++i) {
        const bool in = p.r + i < a.R;
        cp_async_16(dst + i * step, in ? src + i * a.ld : a.x, in);
      }
    }
  } else {
    // copy k of a lane: row k / (tc / 32) of the warp's rows, column lane + 32 (k mod (tc / 32))
    const int lane = threadIdx.x & 31, lp = lg - 3;
    const int64_t r0 = (static_cast<int64_t>(by) << (11 - lg)) + (((threadIdx.x >> 5) << (5 - lg)) << 3);
    const int64_t c0 = (static_cast<int64_t>(bx) << (lg + 2)) + lane;
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const int row = k >> lp, col = 32 * (k & ((1 << lp) - 1));
      const bool in = r0 + row < a.R && c0 + col < a.C;
      cp_async_4(warp_smem + ((row << (lg + 2)) + col + lane) * 4,
                 in ? a.x + (r0 + row) * a.ld + c0 + col : a.x, in);
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncwarp();
}

// The place (16-byte units of BF16, 8-byte units of E4M3 chunks) of a tile column's chunk in
// the shared staging area: in the part of the warp that owns the chunk, the low three bits of
// the column mixed with the chunk index so that the chunk stores of a warp and the column
// reads that follow both spread over the banks.
template <typename CodeT>
__device__ __forceinline__ uint32_t chunk_addr(uint32_t tile_smem, int lg, int col, int chunk) {
  const int sub = chunk & ((1 << (5 - lg)) - 1), w = chunk >> (5 - lg);
  const int pos = (col & ~7) | ((col ^ (col >> 2) ^ chunk) & 7);
  return tile_smem + w * kWarpBytes + (((sub << (lg + 2)) + pos) * 8) * static_cast<int>(sizeof(CodeT));
}

// The transposed copy from the staged chunks: every thread stores 16 bytes (one BF16 chunk or
// two E4M3 chunks) of a tile column at a time.
template <typename CodeT>
__device__ __forceinline__ void store_transposed(const QuantArgs& a, uint32_t tile_smem, unsigned bx,
                                                 unsigned by) {
  constexpr int E = 16 / sizeof(CodeT);   // codes per store
  const int lg = a.lg;
  const int64_t c0 = static_cast<int64_t>(bx) << (lg + 2), r0 = static_cast<int64_t>(by) << (11 - lg);
  __syncthreads();
  if (lg == 5 && a.vec_t && a.pos_rows == nullptr && r0 + 64 <= a.R && c0 + 128 <= a.C) {
    // a whole 64 x 128 tile: a thread's stores are 32 (BF16) or 64 (E4M3) columns apart, its
    // places in the staging area a constant apart
    constexpr int kSpc = sizeof(CodeT) == 2 ? 3 : 2;       // log2(stores per column)
    constexpr int kCols = kQuantThreads >> kSpc;           // columns between a thread's stores
    const int lc = threadIdx.x >> kSpc, st = threadIdx.x & ((1 << kSpc) - 1);
    CodeT* dst = static_cast<CodeT*>(a.codes_t) + (c0 + lc) * a.ldt + r0 + st * E;
    uint32_t from[2];   // of its chunk, or its two chunks
#pragma unroll
    for (int h = 0; h < 16 / (8 * static_cast<int>(sizeof(CodeT))); ++h)
      from[h] = chunk_addr<CodeT>(tile_smem, 5, lc, sizeof(CodeT) == 2 ? st : 2 * st + h);
#pragma unroll
    for (int k = 0; k < 128 / kCols; ++k) {
      uint4 v;
      if constexpr (sizeof(CodeT) == 2) {
        v = ld_shared_v4_u32(from[0] + k * kCols * 16);
      } else {
        const uint2 lo = ld_shared_v2_u32(from[0] + k * kCols * 8), hi = ld_shared_v2_u32(from[1] + k * kCols * 8);
        v = make_uint4(lo.x, lo.y, hi.x, hi.y);
      }
      *reinterpret_cast<uint4*>(dst) = v;
      dst += kCols * a.ldt;
    }
    return;
  }
  if (a.pos_rows != nullptr) {
    // group-ordered: element (column c, row r) goes to pos_rows[r]; a thread keeps its row
    const int lr = 11 - lg;                // log2(rows)
    const int rr = threadIdx.x & ((1 << lr) - 1), step = kQuantThreads >> lr;
    const int64_t r = r0 + rr;
    if (r >= a.R) return;
    int lc = threadIdx.x >> lr;
    const int ncol = static_cast<int>(min(a.C - c0, int64_t(4) << lg));
    CodeT* d = static_cast<CodeT*>(a.codes_t) + (c0 + lc) * a.ldt + ld_here(a.pos_rows + r);
#pragma unroll 4
    for (; lc < ncol; lc += step) {
      *d = ld_shared_code<CodeT>(chunk_addr<CodeT>(tile_smem, lg, lc, rr >> 3) + (rr & 7) * static_cast<int>(sizeof(CodeT)));
      d += step * a.ldt;
    }
    return;
  }
  uint8_t* ct = static_cast<uint8_t*>(a.codes_t);
  const int spc = 8 - lg - (sizeof(CodeT) == 1 ? 1 : 0);   // log2(stores per column)
#pragma unroll 2
  for (int k = 0; k < kTileElems / E / kQuantThreads; ++k) {
    const int idx = threadIdx.x + k * kQuantThreads;
    const int lc = idx >> spc, st = idx & ((1 << spc) - 1);
    const int64_t c = c0 + lc, rs = r0 + st * E;
    if (c >= a.C || rs >= a.R) continue;
    uint4 v;
    if constexpr (sizeof(CodeT) == 2) {
      v = ld_shared_v4_u32(chunk_addr<CodeT>(tile_smem, lg, lc, st));
    } else {
      const uint2 lo = ld_shared_v2_u32(chunk_addr<CodeT>(tile_smem, lg, lc, 2 * st));
      const uint2 hi = ld_shared_v2_u32(chunk_addr<CodeT>(tile_smem, lg, lc, 2 * st + 1));
      v = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
    CodeT* dst = reinterpret_cast<CodeT*>(ct) + c * a.ldt + rs;
    if (a.vec_t && rs + E <= a.R) {
      *reinterpret_cast<uint4*>(dst) = v;
    } else {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (rs + e < a.R)
          dst[e] = static_cast<CodeT>(w[e * sizeof(CodeT) / 4] >> (8 * ((e * sizeof(CodeT)) & 3)));
    }
  }
}

// The values a thread keeps over its rows.
struct QuadState {
  float mul[4], pre[4], cfold[4];   // per column (quad_state)
  unsigned czero;                   // bit j: column j's codes are all 0
  bool merged;                      // (quad_state)
  bool rare;   // inputs quantize to zero for another reason than their value, or need a second scale
  RowValues rv;
  uint64_t state;                   // generator state of element (row, column 0 of the quad)
  TilePos p;
};

// The values of a thread's quad of columns and chunk of rows.  Per column the multiplier (SHIFT:
// 2^e Q / tau_0, where fl(fl(x 2^e) fl(Q / tau_0)) = fl(x (2^e fl(Q / tau_0))) as scaling by 2^e
// is exact -- or, not merged, Q / tau_0 alone with the 2^e in `pre`; PER_COL: Q / range) and the
// folded shift (PER_ROW).  Columns and rows past the last stand for it: their codes are not
// stored.  Everything is loaded before any of it is worked on (the divisions branch, and no load
// moves ahead of a branch): the loads take one latency beside x's, not one after another
// ([3072, 768] transposed weight codes, 4-bit: 4.9 and 4.4 us).
template <int GRAN, int MODE, bool FOLD>
__device__ __forceinline__ QuadState quad_state(const QuantArgs& a, unsigned bx, unsigned by) {
  const float Qf = static_cast<float>(a.Q);
  QuadState t;
  t.p = tile_pos(a.lg, bx, by);
  const int last = static_cast<int>(min(a.C - 1 - t.p.c, int64_t(3)));   // of the quad's columns
  const int64_t c0 = last < 0 ? a.C - 1 : t.p.c;
  const int64_t row = t.p.r + (threadIdx.x & 7), r = min(row, a.R - 1);
  int at[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) at[j] = max(min(j, last), 0);
  uint32_t cexp[4] = {0u, 0u, 0u, 0u}, rexp = 0u, tword = 0u, ftword = 0u;
  float crange[4] = {0.0f, 0.0f, 0.0f, 0.0f}, rrange = 0.0f;
  if (GRAN == SQ_GRAN_SHIFT) {
    tword = a.tslots != nullptr ? slots_word(a.tslots) : __float_as_uint(__ldcg(a.rt));
    load_exponents(a.exp, a.crange, c0, last == 3, at, cexp);
  }
  if (FOLD && a.fold == nullptr) ftword = slots_word(a.ftslots);
  if (GRAN == SQ_GRAN_PER_COL) {
    load_ranges(a.rt + c0, last == 3, at, crange);
    if (FOLD) rexp = load_exponent(a.fold, a.frange, r);
  }
  if (GRAN == SQ_GRAN_PER_ROW) {
    rrange = __ldcg(a.rt + r);
    if (FOLD) load_exponents(a.fold, a.frange, c0, last == 3, at, cexp);
  }

  const float ftau = FOLD && a.fold == nullptr ? slots_tau(ftword) : 0.0f;
  t.rv = {1.0f, 1.0f, 0u};
  t.czero = 0u;
  t.merged = true;
#pragma unroll
  for (int j = 0; j < 4; ++j) t.mul[j] = t.pre[j] = t.cfold[j] = 1.0f;
  const bool write = by == 0 && t.p.chunk == 0;   // the first tiles' columns
  if (GRAN == SQ_GRAN_SHIFT) {
    const float tau = a.tslots != nullptr ? slots_tau(tword) : __uint_as_float(tword);
    const float invS = __fdiv_rn(Qf, tau);
    // tau_0 is 0 or not finite, or Q / tau_0 overflows: every code is 0
    const bool zero = !(tau > 0.0f) || !isfinite(tau) || !isfinite(invS);
    t.merged = isfinite(__fmul_rn(invS, pow2f(a.G - 1)));   // 2^e Q / tau_0 is finite for every e
    t.czero = zero ? 15u : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      cexp[j] = static_cast<uint32_t>(exponent_of(cexp[j], a.exp, tau, a.G));
      t.pre[j] = pow2f(static_cast<int>(cexp[j]));
      t.mul[j] = zero ? 0.0f : (t.merged ? __fmul_rn(invS, t.pre[j]) : invS);
    }
    if (write && a.exp_out != nullptr) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j <= last) a.exp_out[t.p.c + j] = static_cast<uint8_t>(cexp[j]);
    }
    if (bx == 0 && by == 0 && threadIdx.x == 0) {
      *a.scale_out = zero ? 0.0f : __fdiv_rn(tau, Qf);
      if (a.tau_out != nullptr) *a.tau_out = tau;
    }
  }
  if (GRAN == SQ_GRAN_PER_COL) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      bool z = false;
      t.mul[j] = channel_inv(crange[j], Qf, &z);
      t.czero |= z ? 1u << j : 0u;
      if (write && j <= last) a.scale_out[t.p.c + j] = z ? 0.0f : __fdiv_rn(crange[j], Qf);
    }
    if (FOLD) t.rv.fold = pow2f(a.G - 1 - exponent_of(rexp, a.fold, ftau, a.G));
  }
  if (GRAN == SQ_GRAN_PER_ROW) {
    bool z = false;
    t.rv.mul = channel_inv(rrange, Qf, &z);
    z = z && row < a.R;
    t.rv.zero = (__ballot_sync(0xFFFFFFFFu, z) >> (threadIdx.x & 24)) & 0xFFu;
    if (bx == 0 && t.p.col < 32 && row < a.R) a.scale_out[row] = z ? 0.0f : __fdiv_rn(rrange, Qf);
    if (FOLD) {
#pragma unroll
      for (int j = 0; j < 4; ++j) t.cfold[j] = pow2f(a.G - 1 - exponent_of(cexp[j], a.fold, ftau, a.G));
    }
  }
  t.state = 0;   // seed + (idx + 1) gamma
  if (MODE == SQ_ROUND_STOCHASTIC)
    t.state = a.seed + (static_cast<uint64_t>(a.row0 + t.p.r) * static_cast<uint64_t>(a.C) +
                        static_cast<uint64_t>(t.p.c) + 1ull) * kSplitMixGamma;
  t.rare = t.czero != 0u || !t.merged || (GRAN == SQ_GRAN_PER_ROW && t.rv.zero != 0u);
  return t;
}

// The four codes of row i of the quad.
template <typename CodeT, int GRAN, int MODE, bool FOLD>
__device__ __forceinline__ void quantize_quad(const QuadState& t, const float (&x)[4], int i, uint64_t state,
                                              float Qf, uint32_t (&words)[sizeof(CodeT)]) {
  const int src = threadIdx.x & 24;
  const float rmul = GRAN == SQ_GRAN_PER_ROW ? __shfl_sync(0xFFFFFFFFu, t.rv.mul, src | i) : 1.0f;
  const float rfold = GRAN == SQ_GRAN_PER_COL && FOLD ? __shfl_sync(0xFFFFFFFFu, t.rv.fold, src | i) : 1.0f;
  float q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float v = __fmul_rn(x[j], GRAN == SQ_GRAN_PER_ROW ? rmul : t.mul[j]);
    q[j] = MODE == SQ_ROUND_NEAREST_EVEN
               ? round_nearest(v)
               : round_stochastic(v, state + static_cast<uint64_t>(j) * kSplitMixGamma, Qf);
    if (FOLD) q[j] = __fmul_rn(q[j], GRAN == SQ_GRAN_PER_ROW ? t.cfold[j] : rfold);
  }
  encode_words<CodeT, 4>(q, words);
}

template <typename CodeT>
__device__ __forceinline__ CodeT code_of_word(const uint32_t (&words)[sizeof(CodeT)], int j) {
  return static_cast<CodeT>(words[j * sizeof(CodeT) / 4] >> (8 * ((j * sizeof(CodeT)) & 3)));
}

// A row's codes into the thread's slot of that row (where the row of x was, or would be).
template <typename CodeT>
__device__ __forceinline__ void keep_words(uint32_t slot, const uint32_t (&words)[sizeof(CodeT)]) {
  if constexpr (sizeof(CodeT) == 2)
    st_shared_v2(slot, words[0], words[1]);
  else
    st_shared_u32(slot, words[0]);
}

// The chunk of each of the quad's columns -- its code of every row, words[i] those of row i --
// into the staging area.
template <typename CodeT>
__device__ __forceinline__ void stage_chunks(const TilePos& p, int lg, uint32_t tile_smem,
                                             const uint32_t (&words)[8][sizeof(CodeT)]) {
  // (the quad's columns differ in the low two bits of the column alone, which chunk_addr
  // exclusive-ors into the low bits of the place)
  constexpr uint32_t kChunkBytes = 8 * sizeof(CodeT);
  const uint32_t at0 = chunk_addr<CodeT>(tile_smem, lg, p.col, p.chunk);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t to = at0 ^ (j * kChunkBytes);
    if constexpr (sizeof(CodeT) == 2) {
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w[k] = __byte_perm(words[2 * k][j >> 1], words[2 * k + 1][j >> 1], (j & 1) ? 0x7632 : 0x5410);
      st_shared_v4(to, w[0], w[1], w[2], w[3]);
    } else {
      uint32_t w[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t lo = __byte_perm(words[4 * k][0], words[4 * k + 1][0], j | ((4 + j) << 4));
        const uint32_t hi = __byte_perm(words[4 * k + 2][0], words[4 * k + 3][0], j | ((4 + j) << 4));
        w[k] = __byte_perm(lo, hi, 0x5410);
      }
      st_shared_v2(to, w[0], w[1]);
    }
  }
}

// The same from the thread's slots (keep_words), row i's at slot0 + i step.
template <typename CodeT>
__device__ __forceinline__ void stage_slots(const TilePos& p, int lg, uint32_t tile_smem, uint32_t slot0, uint32_t step) {
  uint32_t words[8][sizeof(CodeT)];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if constexpr (sizeof(CodeT) == 2) {
      const uint2 v = ld_shared_v2_u32(slot0 + i * step);
      words[i][0] = v.x;
      words[i][1] = v.y;
    } else {
      words[i][0] = ld_shared_u32(slot0 + i * step);
    }
  }
  __syncwarp();   // every lane's slots have been read: the chunks may overwrite them
  stage_chunks<CodeT>(p, lg, tile_smem, words);
}

// ---------------------------------------------------------------- register path
// What a launch's register path expects of its tensor; tiles that differ take the other path.
enum Form {
  kAligned,   // rows 16-byte aligned in and out
  kShifted,   // rows of x start anywhere
  kOrdered    // aligned rows of x, codes in a group order
};

// Which outputs a kernel writes: the codes, both, the transposed codes alone, or as the arguments
// say.  (Each test in the rows' unrolled body is eight predicated stores more.)
enum Outputs { kCodes, kBoth, kTransposed, kAnyOutputs };

template <int OUT>
__device__ __forceinline__ bool has_codes(const QuantArgs& a) {
  return OUT == kAnyOutputs ? a.codes != nullptr : OUT != kTransposed;
}
template <int OUT>
__device__ __forceinline__ bool has_transposed(const QuantArgs& a) {
  return OUT == kAnyOutputs ? a.codes_t != nullptr : OUT != kCodes;
}

template <int FORM>
__device__ __forceinline__ bool register_tile(const QuantArgs& a, unsigned bx, unsigned by) {
  const int64_t r1 = (static_cast<int64_t>(by) + 1) << (11 - a.lg);
  const int64_t c1 = (static_cast<int64_t>(bx) + 1) << (a.lg + 2);
  if (!a.fast) return false;
  // shifted rows read whole tile rows and up to three elements more: what lies past the last
  // column comes from the following row, which must be there and long enough
  if (FORM == kShifted) return r1 < a.R && c1 + 4 <= a.C + a.ld;
  // aligned tiles may be partial, in whole quads (a group order: whole columns)
  return c1 <= a.C || (FORM == kAligned && (a.C & 3) == 0);
}

// base + i rows of `bytes` bytes, as one multiply-add (a sum of two words would take two
// instructions of the pipe that stochastic rounding fills)
template <typename T>
__device__ __forceinline__ T* row_at(T* base, uint32_t i, uint32_t bytes) {
  uint64_t p;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(p) : "r"(i), "r"(bytes), "l"(base));
  return reinterpret_cast<T*>(p);
}

template <int FORM>
__device__ __forceinline__ void load_registers(const QuantArgs& a, unsigned bx, unsigned by, float4 (&x)[8]) {
  const TilePos p = tile_pos(a.lg, bx, by);
  if (FORM != kShifted) {
    // quads and rows outside the tensor read its first column and its last row: their codes are
    // not stored
    const float* src = a.x + (p.c < a.C ? p.c : 0);
    if (p.r + 8 <= a.R) {
      src += p.r * a.ld;
      const uint32_t row = static_cast<uint32_t>(a.ld * 4);
      if (a.sectors) {   // (set_alignment)
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = ld_stream_v4(row_at(src, i, row));
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = ld_rows_v4(row_at(src, i, row));
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = ld_stream_v4(src + min(p.r + i, a.R - 1) * a.ld);
    }
    return;
  }
  // Of each row the lanes read the aligned vectors that cover the tile, and each takes the
  // elements past its own vector from its neighbour -- the last lane of a row from the vector
  // after the tile, which lane i of the row's lanes reads for row i.
  const int lane = threadIdx.x & 31, lpr = 1 << a.lg;   // lanes per row
  const int64_t off = p.r * a.ld + p.c;
  const bool last = (lane & (lpr - 1)) == lpr - 1;
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = ld_stream_v4(a.x + ((off + i * a.ld) & ~int64_t(3)));
  const float4 e = ld_stream_v4(a.x + ((off - p.col + lpr * 4 + (lane & 7) * a.ld) & ~int64_t(3)));
  const int grp = lane & ~(lpr - 1);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int sh = static_cast<int>((off + i * a.ld) & 3);   // the same for all lanes of a row
    const float4 v = x[i];
    float4 n;
    n.x = __shfl_down_sync(0xFFFFFFFFu, v.x, 1);
    n.y = __shfl_down_sync(0xFFFFFFFFu, v.y, 1);
    n.z = __shfl_down_sync(0xFFFFFFFFu, v.z, 1);
    const float ex = __shfl_sync(0xFFFFFFFFu, e.x, grp | i);
    const float ey = __shfl_sync(0xFFFFFFFFu, e.y, grp | i);
    const float ez = __shfl_sync(0xFFFFFFFFu, e.z, grp | i);
    if (last) {
      n.x = ex;
      n.y = ey;
      n.z = ez;
    }
    if (sh == 1) x[i] = make_float4(v.y, v.z, v.w, n.x);
    if (sh == 2) x[i] = make_float4(v.z, v.w, n.x, n.y);
    if (sh == 3) x[i] = make_float4(v.w, n.x, n.y, n.z);
  }
}

template <typename CodeT, int FORM, int GRAN, int MODE, bool FOLD, int OUT>
__device__ __forceinline__ void quantize_registers(const QuantArgs& a, const QuadState& t, const float4 (&xin)[8],
                                                   uint32_t tile_smem) {
  const float Qf = static_cast<float>(a.Q);
  const uint64_t row_step = static_cast<uint64_t>(a.C) * kSplitMixGamma;
  const bool ordered = FORM == kOrdered && OUT != kTransposed && a.pos_cols != nullptr;
  CodeT* const first = static_cast<CodeT*>(a.codes) + t.p.r * a.ldc + t.p.c;
  const uint32_t row = static_cast<uint32_t>(a.ldc * static_cast<int64_t>(sizeof(CodeT)));
  // the codes are kept in the thread's slots for the transposed copy and for a group order
  const bool trans = has_transposed<OUT>(a);
  constexpr bool kHeld = OUT == kTransposed;   // nothing else to keep in registers: no slots
  const bool kept = !kHeld && (trans || ordered);
  uint32_t held[kHeld ? 8 : 1][sizeof(CodeT)];
  const uint32_t warp_smem = tile_smem + (threadIdx.x >> 5) * kWarpBytes;
  uint64_t state = t.state;
  // (slots of four codes each, those of a row side by side: no two lanes' stores share a bank)
  constexpr uint32_t kSlot = 4 * sizeof(CodeT);
  const uint32_t keep = warp_smem + (quad_slot(0, a.lg, 0) >> 4) * kSlot, step = kSlot << a.lg;
  // rows of the quad to store
  const int rows = !has_codes<OUT>(a) || ordered || t.p.c >= a.C ? 0 : static_cast<int>(min(a.R - t.p.r, int64_t(8)));
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float x[4] = {xin[i].x, xin[i].y, xin[i].z, xin[i].w};
    uint32_t words[sizeof(CodeT)];
    quantize_quad<CodeT, GRAN, MODE, FOLD>(t, x, i, state, Qf, words);
    state += row_step;
    if (i < rows) {
      CodeT* dst = row_at(first, i, row);
      if (FORM == kShifted && t.p.c + 3 >= a.C) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (t.p.c + j < a.C) dst[j] = code_of_word<CodeT>(words, j);
      } else if constexpr (sizeof(CodeT) == 2) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[1]);
      } else {
        *reinterpret_cast<uint32_t*>(dst) = words[0];
      }
    }
    if (kept) keep_words<CodeT>(keep + i * step, words);
    if constexpr (kHeld) {
#pragma unroll
      for (int k = 0; k < static_cast<int>(sizeof(CodeT)); ++k) held[i][k] = words[k];
    }
  }
  if (ordered) {
    // The channels of a group keep their order, so 32 consecutive columns go to a few runs of
    // consecutive places: one column a lane writes whole runs, where a lane's own four columns
    // would write two bytes of every eight (four times the partial sectors).
    const int lane = threadIdx.x & 31, groups = 1 << (a.lg - 3);   // of 32 columns in the tile
    const int64_t cb = t.p.c - t.p.col + lane, rb = t.p.r - 8 * (lane >> a.lg);   // the warp's first row
    int at[4];
#pragma unroll
    for (int g = 0; g < 4; ++g)
      if (g < groups) at[g] = ld_here(a.pos_cols + cb + 32 * g);
    const int nrows = static_cast<int>(min(a.R - rb, int64_t(64 >> (a.lg - 2))));
    // (column 32 g + lane of the warp's row r)
    uint32_t from = warp_smem + lane * static_cast<int>(sizeof(CodeT));
    CodeT* d = static_cast<CodeT*>(a.codes) + rb * a.ldc;
    __syncwarp();
#pragma unroll 2
    for (int r = 0; r < nrows; ++r) {
#pragma unroll
      for (int g = 0; g < 4; ++g)
        if (g < groups) d[at[g]] = ld_shared_code<CodeT>(from + g * 32 * static_cast<int>(sizeof(CodeT)));
      from += step;
      d += a.ldc;
    }
    __syncwarp();   // the chunks may overwrite the slots
  }
  if constexpr (kHeld)
    stage_chunks<CodeT>(t.p, a.lg, tile_smem, held);
  else if (trans)
    stage_slots<CodeT>(t.p, a.lg, tile_smem, keep, step);
}

// ------------------------------------------------------------ shared-memory path
template <typename CodeT, int GRAN, int MODE, bool FOLD>
__device__ __forceinline__ void quantize_rows(const QuantArgs& a, const QuadState& t, uint32_t tile_smem) {
  const float Qf = static_cast<float>(a.Q);
  const uint32_t slot0 = quad_slot(tile_smem + (threadIdx.x >> 5) * kWarpBytes, a.lg, 0), step = 16u << a.lg;
  const uint64_t row_step = static_cast<uint64_t>(a.C) * kSplitMixGamma;
  uint64_t state = t.state;
  const int rows = static_cast<int>(a.R - t.p.r < 8 ? (a.R - t.p.r < 0 ? 0 : a.R - t.p.r) : 8);
  // four codes in one store; otherwise the place of each column's code in a row (-1: none)
  const bool wide = a.vec_out && a.pos_cols == nullptr && t.p.c + 3 < a.C;
  int64_t at[4] = {-1, -1, -1, -1};
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (a.codes != nullptr && !wide && t.p.c + j < a.C)
      at[j] = a.pos_cols != nullptr ? ld_here(a.pos_cols + t.p.c + j) : t.p.c + j;
  CodeT* dst = static_cast<CodeT*>(a.codes) + t.p.r * a.ldc + (wide ? t.p.c : 0);
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    const uint32_t slot = slot0 + i * step;
    const float4 x4 = ld_shared_v4_f32(slot);
    float x[4] = {x4.x, x4.y, x4.z, x4.w};
    if (t.rare) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (GRAN == SQ_GRAN_SHIFT && !t.merged) x[j] = __fmul_rn(x[j], t.pre[j]);
        if (((t.czero >> j) & 1u) || (GRAN == SQ_GRAN_PER_ROW && ((t.rv.zero >> i) & 1u))) x[j] = 0.0f;
      }
    }
    uint32_t words[sizeof(CodeT)];
    quantize_quad<CodeT, GRAN, MODE, FOLD>(t, x, i, state, Qf, words);
    state += row_step;
    if (a.codes != nullptr && i < rows) {
      if (wide) {
        if constexpr (sizeof(CodeT) == 2)
          *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[1]);
        else
          *reinterpret_cast<uint32_t*>(dst) = words[0];
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (at[j] >= 0) dst[at[j]] = code_of_word<CodeT>(words, j);
      }
      dst += a.ldc;
    }
    if (a.codes_t != nullptr) keep_words<CodeT>(slot, words);
  }
  if (a.codes_t != nullptr) stage_slots<CodeT>(t.p, a.lg, tile_smem, slot0, step);
}

// One tile of a tensor.
// WAIT: x may be read before the preceding kernel has completed (it did not write x), its
// results only after the wait.
template <typename CodeT, int FORM, int GRAN, int MODE, bool FOLD, int OUT, bool WAIT = false>
__device__ __forceinline__ void quantize_block(const QuantArgs& a, unsigned bx, unsigned by, uint32_t tile_smem) {
  bool fast = register_tile<FORM>(a, bx, by);
  float4 x[8];
  if (fast) load_registers<FORM>(a, bx, by, x);
  if (WAIT) griddep_wait();
  const QuadState t = quad_state<GRAN, MODE, FOLD>(a, bx, by);
  fast = fast && !__any_sync(0xFFFFFFFFu, t.rare);   // (each warp by itself: their parts of the tile are their own)
  if (fast) {
    quantize_registers<CodeT, FORM, GRAN, MODE, FOLD, OUT>(a, t, x, tile_smem);
  } else {
    load_tile(a, bx, by, tile_smem + (threadIdx.x >> 5) * kWarpBytes);
    quantize_rows<CodeT, GRAN, MODE, FOLD>(a, t, tile_smem);
  }
  if (has_transposed<OUT>(a)) store_transposed<CodeT>(a, tile_smem, bx, by);
}

template <typename CodeT, int FORM, int GRAN, int MODE, bool FOLD, int OUT>
__global__ void __launch_bounds__(kQuantThreads, 4) quantize_kernel(const QuantArgs a) {
  __shared__ __align__(128) uint8_t tile[8 * kWarpBytes];
  // launched early behind the range pass: nothing it wrote (nor x) is read before it is done
  if (!a.beside) griddep_wait();
  griddep_launch_dependents();
  quantize_block<CodeT, FORM, GRAN, MODE, FOLD, OUT>(a, blockIdx.x, blockIdx.y, smem_u32(tile));
  if (a.beside) griddep_wait();
}

template <typename CodeT, int FORM, int GRAN, int MODE, bool FOLD, int OUT>
static void launch_outputs(const QuantArgs& a, dim3 grid, cudaStream_t s) {
  launch_pdl(quantize_kernel<CodeT, FORM, GRAN, MODE, FOLD, OUT>, grid, dim3(kQuantThreads), s, a);
}

// The outputs that get a kernel of their own: ShiftQuant's codes with and without the copy, and
// what each role of a weight writes.
template <typename CodeT, int FORM, int GRAN, int MODE, bool FOLD>
static void launch_form(const QuantArgs& a, dim3 grid, cudaStream_t s) {
  constexpr bool kShift = GRAN == SQ_GRAN_SHIFT, kWeight = !kShift && MODE == SQ_ROUND_NEAREST_EVEN;
  if constexpr (kShift) {
    if (a.codes != nullptr && a.codes_t != nullptr)
      return launch_outputs<CodeT, FORM, GRAN, MODE, FOLD, kBoth>(a, grid, s);
  }
  if constexpr (kShift || (kWeight && GRAN == SQ_GRAN_PER_ROW)) {
    if (a.codes_t == nullptr) return launch_outputs<CodeT, FORM, GRAN, MODE, FOLD, kCodes>(a, grid, s);
  }
  if constexpr (kWeight && GRAN == SQ_GRAN_PER_COL) {
    if (a.codes == nullptr) return launch_outputs<CodeT, FORM, GRAN, MODE, FOLD, kTransposed>(a, grid, s);
  }
  launch_outputs<CodeT, FORM, GRAN, MODE, FOLD, kAnyOutputs>(a, grid, s);
}

template <typename CodeT, int FORM, int GRAN, bool FOLD>
static void launch_mode(const QuantArgs& a, int mode, dim3 grid, cudaStream_t s) {
  if (mode == SQ_ROUND_NEAREST_EVEN)
    launch_form<CodeT, FORM, GRAN, SQ_ROUND_NEAREST_EVEN, FOLD>(a, grid, s);
  else
    launch_form<CodeT, FORM, GRAN, SQ_ROUND_STOCHASTIC, FOLD>(a, grid, s);
}

template <typename CodeT, int FORM>
static void launch_gran(const QuantArgs& a, int gran, int mode, dim3 grid, cudaStream_t s) {
  const bool fold = FORM != kOrdered && (a.fold != nullptr || a.frange != nullptr);   // group-ordered codes carry no fold
  if (gran == SQ_GRAN_SHIFT) {
    launch_mode<CodeT, FORM, SQ_GRAN_SHIFT, false>(a, mode, grid, s);
  } else if (gran == SQ_GRAN_PER_COL) {
    if (fold) launch_mode<CodeT, FORM, SQ_GRAN_PER_COL, FORM != kOrdered>(a, mode, grid, s);
    else launch_mode<CodeT, FORM, SQ_GRAN_PER_COL, false>(a, mode, grid, s);
  } else {
    if (fold) launch_mode<CodeT, FORM, SQ_GRAN_PER_ROW, FORM != kOrdered>(a, mode, grid, s);
    else launch_mode<CodeT, FORM, SQ_GRAN_PER_ROW, false>(a, mode, grid, s);
  }
}

template <typename CodeT>
static void launch_quantize(const QuantArgs& a, int gran, int mode, dim3 grid, cudaStream_t s) {
  switch (a.form) {
    case kAligned: launch_gran<CodeT, kAligned>(a, gran, mode, grid, s); break;
    case kShifted: launch_gran<CodeT, kShifted>(a, gran, mode, grid, s); break;
    default: launch_gran<CodeT, kOrdered>(a, gran, mode, grid, s); break;
  }
}

// Both roles of a weight from one pass over it (Sec. 5.1): the forward GEMM's
// per-out-channel codes (gran PER_COL, written transposed, the fold indexed by row) and loss
// propagation's per-in-channel codes (gran PER_ROW, natural layout, the fold indexed by
// column), both from one load of the block's tile, held in registers (in shared memory on the
// general path).  Bound by HBM with four blocks an SM: a [4096, 11008] weight, 8-bit, takes 63.5
// us, of which 42.8 for the transposed codes alone and 40.2 for the others.
template <typename CodeT, int FORM, bool FF, bool FD, bool WAIT = false>
__device__ __forceinline__ void quantize_weight_block(const QuantArgs& af, const QuantArgs& ad, unsigned bx,
                                                      unsigned by, uint32_t tile_smem) {
  // both roles read the same tensor: af and ad share x, R, C, ld, lg
  constexpr int kCol = SQ_GRAN_PER_COL, kRow = SQ_GRAN_PER_ROW, kRn = SQ_ROUND_NEAREST_EVEN;
  bool fast = register_tile<FORM>(af, bx, by) && register_tile<FORM>(ad, bx, by);
  float4 x[8];
  if (fast) load_registers<FORM>(af, bx, by, x);
  if (WAIT) griddep_wait();
  const QuadState td = quad_state<kRow, kRn, FD>(ad, bx, by);
  fast = fast && !__any_sync(0xFFFFFFFFu, td.rare);
  if (fast) {
    quantize_registers<CodeT, FORM, kRow, kRn, FD, kCodes>(ad, td, x, tile_smem);
  } else {   // the per-in-channel role has no transposed copy: it leaves the tile as it is
    load_tile(af, bx, by, tile_smem + (threadIdx.x >> 5) * kWarpBytes);
    quantize_rows<CodeT, kRow, kRn, FD>(ad, td, tile_smem);
  }
  const QuadState tf = quad_state<kCol, kRn, FF>(af, bx, by);
  if (fast && __any_sync(0xFFFFFFFFu, tf.rare)) {
    load_tile(af, bx, by, tile_smem + (threadIdx.x >> 5) * kWarpBytes);
    fast = false;
  }
  if (fast)
    quantize_registers<CodeT, FORM, kCol, kRn, FF, kTransposed>(af, tf, x, tile_smem);
  else
    quantize_rows<CodeT, kCol, kRn, FF>(af, tf, tile_smem);
  store_transposed<CodeT>(af, tile_smem, bx, by);
}

template <typename CodeT, int FORM, bool FF, bool FD>
__global__ void __launch_bounds__(kQuantThreads, 4) quantize_weight_kernel(const QuantArgs af, const QuantArgs ad) {
  __shared__ __align__(128) uint8_t tile[8 * kWarpBytes];
  if (!af.beside) griddep_wait();
  griddep_launch_dependents();
  quantize_weight_block<CodeT, FORM, FF, FD>(af, ad, blockIdx.x, blockIdx.y, smem_u32(tile));
  if (af.beside) griddep_wait();
}

template <typename CodeT, int FORM>
static void launch_weight_folds(const QuantArgs& af, const QuantArgs& ad, dim3 grid, cudaStream_t s) {
  const bool ff = af.fold != nullptr || af.frange != nullptr, fd = ad.fold != nullptr || ad.frange != nullptr;
  const dim3 block(kQuantThreads);
  if (ff && fd) launch_pdl(quantize_weight_kernel<CodeT, FORM, true, true>, grid, block, s, af, ad);
  else if (ff) launch_pdl(quantize_weight_kernel<CodeT, FORM, true, false>, grid, block, s, af, ad);
  else if (fd) launch_pdl(quantize_weight_kernel<CodeT, FORM, false, true>, grid, block, s, af, ad);
  else launch_pdl(quantize_weight_kernel<CodeT, FORM, false, false>, grid, block, s, af, ad);
}

template <typename CodeT>
static void launch_quantize_weight(const QuantArgs& af, const QuantArgs& ad, dim3 grid, cudaStream_t s) {
  if (af.form == kShifted)
    launch_weight_folds<CodeT, kShifted>(af, ad, grid, s);
  else
    launch_weight_folds<CodeT, kAligned>(af, ad, grid, s);
}

// ============================================================= a layer's quantizer passes
// The quantizer passes of a layer step (X, dY and W: three tensors, eleven launches one by
// one, each short next to its launch gap and its last wave) as one launch each: the
// accumulators zeroed, every tensor's range pass, every tensor's codes (three launches beside one
// another for large layers).  The grouping needs no launch of its own: the range pass also keeps
// tau_0 (kTauSlots words per tensor), and a quantizer block forms the exponents of its own
// columns, and the shifts it folds into weight codes, from the ranges and tau_0.
//
// What a launch of this chain may rely on.  Each is launched behind the one before it and starts
// when every block of that one has let it (griddep_launch_dependents) or has ended:
//   layer_init     waits for whatever precedes it, only then lets the range pass start -- so x,
//                  dy and w are complete when that starts, and it reads them before its own wait;
//   layer_range    waits (for the zeroed accumulators) before its first atomic, and lets the codes
//                  start after that wait;
//   codes, first   layer_quantize loads x early and waits before anything the range pass wrote;
//                  quantize_kernel of X waits first, and only then lets the next one start;
//   codes, beside  those of W and dY read x, ranges and tau_0 (past L1) without a wait: the launch
//                  before them was let go by one that had waited for the range pass.  Their wait
//                  comes last, so that whoever waits for dY's launch has waited for all three;
//   GEMM           waits before everything.
// A kernel put between two of these must wait before it lets the next one start, and a launch
// that writes x, dy, w or the ranges must not come after layer_init.
struct LayerInit {
  unsigned* p[5];
  int64_t n[5];
};

// The first of the three, launched behind whatever precedes it: it waits for that before it
// writes, and lets the range pass launch only then.
__global__ void __launch_bounds__(256) layer_init_kernel(const LayerInit z) {
  griddep_wait();
  griddep_launch_dependents();
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
#pragma unroll
  for (int k = 0; k < 5; ++k)
    for (int64_t i = i0; i < z.n[k]; i += stride) z.p[k][i] = 0u;
}

constexpr int kZeroVecs = 2048;   // 16-byte words a zeroing block clears
constexpr int kZeroRegions = 3;

struct LayerRange {
  RangeView w, g, x;
  int wrun;                       // column blocks a weight block walks
  int glg, xlg;
  unsigned wgx, ggx, xgx;         // blocks across the columns
  unsigned zend, wend, gend;      // first block past the zeroing, W's and dY's blocks
  uint4* zero[kZeroRegions];      // regions the layer's GEMMs want zeroed
  int64_t zvecs[kZeroRegions];    // in 16-byte words
  unsigned zblocks[kZeroRegions];
  unsigned *wcols, *wrows, *gcols, *xcols, *gtau, *xtau;
  int* status;
};

// one tile of a ShiftQuant tensor: column maxima and their largest to a tau_0 slot.  An atomic
// goes out only where it would raise the value seen.
template <int FORM>
__device__ __forceinline__ void layer_range_tile(const RangeView& v, int lg, unsigned bx, unsigned by, unsigned* red,
                                                 unsigned* cols, unsigned* tau, int* status) {
  const int tid = threadIdx.x;
  const int tc = 4 << lg, rpp = (kColTx * kColTy) >> lg;
  const int qc = tid & ((1 << lg) - 1), ro = tid >> lg;
  const int64_t cb = static_cast<int64_t>(bx) * tc;
  unsigned m[4] = {0u, 0u, 0u, 0u}, rm[8];
  tile_maxima<false, FORM>(v, lg, cb, static_cast<int64_t>(by) * 8 * rpp + ro, qc, m, rm);
  put_maxima<FORM>(red, lg, ro, qc, m);
  __syncthreads();
  griddep_wait();   // the accumulators are zero
  griddep_launch_dependents();
  if (tid >= 128) return;
  unsigned w = 0u;
  const int64_t c = cb + tid;
  if (tid < tc && c < v.C) {
    w = get_maximum(red, lg, tid);
    unsigned* p = column_bits<FORM>(cols, v, c);
    if (w > __ldcg(p)) atomicMax(p, w);
  }
  w = __reduce_max_sync(0xFFFFFFFFu, w);
  if ((tid & 31) == 0) {
    unsigned* p = tau + (bx + by) % kTauSlots;
    if (w > __ldcg(p)) atomicMax(p, w);
    if (w >= 0x7F800000u) atomicOr(status, kDevNonFinite);
  }
}

// a tile of whichever form the tensor has; PLAIN: all three are kViewVec
template <bool PLAIN>
__device__ __forceinline__ void layer_range_any(const RangeView& v, int lg, unsigned gx, unsigned b, unsigned* red,
                                                unsigned* cols, unsigned* tau, int* status) {
  if (PLAIN || v.form == kViewVec)
    layer_range_tile<kViewVec>(v, lg, b % gx, b / gx, red, cols, tau, status);
  else if (v.form == kViewFolded)
    layer_range_tile<kViewFolded>(v, lg, b % gx, b / gx, red, cols, tau, status);
  else
    layer_range_tile<kViewStrided>(v, lg, b % gx, b / gx, red, cols, tau, status);
}

template <bool PLAIN>
__global__ void __launch_bounds__(256, 4) layer_range_kernel(const LayerRange a) {
  __shared__ unsigned red[kColTy * kColTx * 4];
  unsigned b = blockIdx.x;
  if (b < a.zend) {
    // (the preceding GEMM may still read these until the first kernel has waited for it)
    griddep_wait();
    griddep_launch_dependents();
    int k = 0;
    while (k + 1 < kZeroRegions && b >= a.zblocks[k]) b -= a.zblocks[k++];
    const int64_t end = min(a.zvecs[k], (static_cast<int64_t>(b) + 1) * kZeroVecs);
    for (int64_t i = static_cast<int64_t>(b) * kZeroVecs + threadIdx.x; i < end; i += 256)
      a.zero[k][i] = make_uint4(0u, 0u, 0u, 0u);
  } else if (b < a.wend) {
    b -= a.zend;
    bool bad = false;
    if (PLAIN || a.w.form == kViewVec)
      weight_range_run<kViewVec>(a.w, b / a.wgx, static_cast<int64_t>(b % a.wgx) * a.wrun, a.wrun, red, a.wcols,
                                 a.wrows, &bad);
    else
      weight_range_run<kViewStrided>(a.w, b / a.wgx, static_cast<int64_t>(b % a.wgx) * a.wrun, a.wrun, red, a.wcols,
                                     a.wrows, &bad);
    griddep_launch_dependents();
    if (bad) atomicOr(a.status, kDevNonFinite);
  } else if (b < a.gend) {
    b -= a.wend;
    layer_range_any<PLAIN>(a.g, a.glg, a.ggx, b, red, a.gcols, a.gtau, a.status);
  } else {
    b -= a.gend;
    layer_range_any<PLAIN>(a.x, a.xlg, a.xgx, b, red, a.xcols, a.xtau, a.status);
  }
}

// The blocks of X, W and dY one list after another: X was the last tensor of the range pass,
// so as much of it as fits is still in L2.
struct LayerQuant {
  QuantArgs x, g, wf, wd;
  unsigned xgx, ggx, wgx;
  unsigned xend, wend;   // first block past X's and W's
};

template <typename CodeT, int FORM>
__global__ void __launch_bounds__(kQuantThreads, 4) layer_quantize_kernel(const LayerQuant q) {
  __shared__ __align__(128) uint8_t tile[8 * kWarpBytes];
  const uint32_t smem = smem_u32(tile);
  griddep_launch_dependents();
  unsigned b = blockIdx.x;
  if (b < q.xend) {
    quantize_block<CodeT, FORM, SQ_GRAN_SHIFT, SQ_ROUND_NEAREST_EVEN, false, kAnyOutputs, true>(q.x, b % q.xgx, b / q.xgx, smem);
  } else if (b < q.wend) {
    b -= q.xend;
    quantize_weight_block<CodeT, FORM, true, true, true>(q.wf, q.wd, b % q.wgx, b / q.wgx, smem);
  } else {
    b -= q.wend;
    quantize_block<CodeT, FORM, SQ_GRAN_SHIFT, SQ_ROUND_STOCHASTIC, false, kAnyOutputs, true>(q.g, b % q.ggx, b / q.ggx, smem);
  }
}

// ============================================================ group order (Sec. 3.2)
// The inner index of a forward or loss-propagation GEMM in group order: every group's
// channels contiguous (stable: in channel order within a group), each group's segment
// starting on a K-block boundary (bk elements), so that the contraction can accumulate a
// group unshifted and apply its shift once per segment.  seg[0..G] = segment starts (seg[G]
// = the padded width), seg[G+1..2G] = channels per group; pos[c] = the position of channel
// c.  One block: counts per group, then stable ranks chunk by chunk with warp ballots.
constexpr int kOrderThreads = 1024;

__global__ void __launch_bounds__(kOrderThreads)
    group_order_kernel(const uint8_t* __restrict__ exp, int64_t C, int G, int bk,
                       int* __restrict__ pos, int* __restrict__ seg) {
  __shared__ int cnt[8];
  __shared__ int start[9];
  __shared__ int base[8];
  __shared__ int wtot[kOrderThreads / 32][8];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid < 8) cnt[tid] = 0;
  __syncthreads();
  int mine[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t c = tid; c < C; c += kOrderThreads) {
    const int e = min(static_cast<int>(exp[c]), G - 1);
#pragma unroll
    for (int g = 0; g < 8; ++g) mine[g] += (e == g);
  }
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    const int v = __reduce_add_sync(0xFFFFFFFFu, mine[g]);
    if (lane == 0 && v) atomicAdd(&cnt[g], v);
  }
  __syncthreads();
  if (tid == 0) {
    int o = 0;
    for (int g = 0; g < G; ++g) {
      start[g] = o;
      o += (cnt[g] + bk - 1) / bk * bk;
      base[g] = 0;
    }
    start[G] = o;
    for (int g = 0; g <= G; ++g) seg[g] = start[g];
    for (int g = 0; g < G; ++g) seg[G + 1 + g] = cnt[g];
  }
  __syncthreads();
  for (int64_t c0 = 0; c0 < C; c0 += kOrderThreads) {
    const int64_t c = c0 + tid;
    const int e = c < C ? min(static_cast<int>(exp[c]), G - 1) : -1;
    const unsigned below = (1u << lane) - 1u;
    int rank = 0;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const unsigned b = __ballot_sync(0xFFFFFFFFu, e == g);
      if (e == g) rank = __popc(b & below);
      if (lane == 0) wtot[w][g] = __popc(b);
    }
    __syncthreads();
    if (e >= 0) {
      int before = 0;
      for (int k = 0; k < w; ++k) before += wtot[k][e];
      pos[c] = start[e] + base[e] + before + rank;
    }
    __syncthreads();
    if (tid < G) {
      int t = 0;
      for (int k = 0; k < kOrderThreads / 32; ++k) t += wtot[k][tid];
      base[tid] += t;
    }
    __syncthreads();
  }
}

// zero the padding positions of a group-ordered code buffer [rows, ld]: the tail
// [seg[g] + count_g, seg[g+1]) of every segment, one warp per row
template <typename CodeT>
__global__ void __launch_bounds__(256)
    order_pad_kernel(CodeT* __restrict__ codes, int64_t rows, int64_t ld, const int* __restrict__ seg,
                     int G) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) / 32; r < rows;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x / 32) {
    CodeT* row = codes + r * ld;
    for (int g = 0; g < G; ++g) {
      const int from = seg[g] + seg[G + 1 + g], to = seg[g + 1];
      for (int i = from + lane; i < to; i += 32) row[i] = CodeT(0);
    }
  }
}

// How the range pass reads x [rows, cols].  Folding applies to dense unaligned tensors; a
// weight's row maxima need its own rows (fold = false).
static RangeView range_view(const float* x, int64_t rows, int64_t cols, int64_t ld, bool fold) {
  RangeView v = {x, rows, cols, ld, (ld % 4 == 0) && aligned16(x) ? kViewVec : kViewStrided, cols, 0};
  const int64_t f = cols % 2 == 0 ? 2 : 4;   // rows that make a multiple of four elements
  if (v.form == kViewStrided && fold && ld == cols && aligned16(x) && rows >= f) {
    v.R = rows / f;
    v.C = v.ld = f * cols;
    v.form = kViewFolded;
    v.tail = (rows - v.R * f) * cols;
  }
  return v;
}

// log2 of a quarter of the range pass's tile width: the column count rounded up to a power of
// two, 4 to 128
static int range_lg(int64_t cols) {
  int lg = 0;
  while (lg < 5 && (int64_t(4) << lg) < cols) ++lg;
  return lg;
}

// The range pass of x [rows, cols] (0 < rows, 0 < cols < 2^36, checked by the callers):
// one block per tile, narrow tensors in whole clusters along the rows; with
// row_bits also the per-row maxima.
static cudaError_t launch_range(const float* x, int64_t rows, int64_t cols, int64_t ld,
                                unsigned* col_bits, unsigned* row_bits, int* status,
                                cudaStream_t s) {
  const RangeView v = range_view(x, rows, cols, ld, row_bits == nullptr);
  // a weight's row ranges need whole 128-column warp rows
  const int lg = row_bits != nullptr ? 5 : range_lg(v.C);
  const int64_t tc = int64_t(4) << lg;
  const int64_t cblocks = (v.C + tc - 1) / tc;   // < 2^31: C < 2^38, tc = 128 past 64
  const int64_t tiles = (v.R + 8 * (256 >> lg) - 1) / (8 * (256 >> lg));
  const int cl = cols <= kRangeClusterMaxCols ? kRangeCluster : 1;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.blockDim = dim3(kColTx, kColTy);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t err;
  if (row_bits != nullptr && cl == 1) {
    // a wide weight: runs of column blocks per block (weight_range_kernel)
    const int64_t runs = (cblocks + kWeightRun - 1) / kWeightRun;
    cfg.gridDim = dim3(static_cast<unsigned>(runs), static_cast<unsigned>(tiles < 65535 ? tiles : 65535));
    err = cudaLaunchKernelEx(&cfg, v.form == kViewVec ? weight_range_kernel<kViewVec> : weight_range_kernel<kViewStrided>, v,
                             col_bits, row_bits, status);
    if (err == cudaSuccess) err = cudaGetLastError();
    return err;
  }
  const int64_t max_rblocks = 65535 / cl * cl;
  int64_t rblocks = (tiles + cl - 1) / cl * cl;
  if (rblocks > max_rblocks) rblocks = max_rblocks;
  cfg.gridDim = dim3(static_cast<unsigned>(cblocks), static_cast<unsigned>(rblocks));
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = cl;
  attr[1].val.clusterDim.z = 1;
  cfg.numAttrs = cl > 1 ? 2 : 1;
  auto kernel = row_bits != nullptr   // a narrow weight (wide ones returned above)
                    ? (v.form == kViewVec ? colmax_kernel<kRangeCluster, true, kViewVec>
                                          : colmax_kernel<kRangeCluster, true, kViewStrided>)
                : cl > 1 ? (v.form == kViewVec      ? colmax_kernel<kRangeCluster, false, kViewVec>
                            : v.form == kViewFolded ? colmax_kernel<kRangeCluster, false, kViewFolded>
                                                    : colmax_kernel<kRangeCluster, false, kViewStrided>)
                         : (v.form == kViewVec      ? colmax_kernel<1, false, kViewVec>
                            : v.form == kViewFolded ? colmax_kernel<1, false, kViewFolded>
                                                    : colmax_kernel<1, false, kViewStrided>);
  err = cudaLaunchKernelEx(&cfg, kernel, v, lg, col_bits, row_bits, status);
  if (err == cudaSuccess) err = cudaGetLastError();
  return err;
}

// the sizes one quantizer launch takes (64-row tiles in a grid's 65535 rows)
static bool quant_grid_ok(int64_t rows, int64_t cols) {
  return (cols + 127) / 128 <= 0x7FFFFFFF && (rows + 63) / 64 <= 65535;
}

static dim3 quant_grid(const QuantArgs& a) {
  return dim3(static_cast<unsigned>((a.C + tile_cols(a.lg) - 1) / tile_cols(a.lg)),
              static_cast<unsigned>((a.R + tile_rows(a.lg) - 1) / tile_rows(a.lg)));
}

// alignment of the tensor and its outputs (given with their group orders), and from it the
// form of the launch's register path
static void set_alignment(QuantArgs* a, int cbytes) {
  a->vec_in = aligned16(a->x) && a->ld % 4 == 0;
  // Rows that start inside a sector share it with the row or the tile before, and are read
  // through L1 (8-bit codes, round to nearest, 30 million elements, past L1 / through it: 292
  // columns 37.5 / 30.8 us, 420 columns 36.0 / 30.0 us).  Rows of whole sectors are not: there is
  // nothing to share, and the quantizer passes of a layer step, whose x is in L2, take 1-4 us more.
  a->sectors = reinterpret_cast<uintptr_t>(a->x) % 32 == 0 && a->ld % 8 == 0;
  a->vec_out = a->codes != nullptr && a->ldc % 4 == 0 && reinterpret_cast<uintptr_t>(a->codes) % (4 * cbytes) == 0;
  a->vec_t = a->codes_t != nullptr && (a->ldt * cbytes) % 16 == 0 && aligned16(a->codes_t);
  a->lg = tile_lg(a->C);
  const bool ordered = a->pos_cols != nullptr || a->pos_rows != nullptr;
  a->form = ordered ? kOrdered : (a->vec_in ? kAligned : kShifted);
  const bool in = a->form == kShifted ? aligned16(a->x) : a->vec_in != 0;
  // (rows of less than 4 GB: row_at)
  a->fast = in && (a->codes == nullptr || a->vec_out || a->pos_cols != nullptr) && a->ld < (int64_t(1) << 30) &&
            a->ldc < (int64_t(1) << 31);
}

// both roles of a weight (the folds are set by the caller)
static void weight_args(QuantArgs* af, QuantArgs* ad, const float* w, int64_t rows, int64_t cols, int64_t ld,
                        int bits, int n_groups, const float* range_out_ch, const float* range_in_ch,
                        void* codes_fwd, int64_t ld_fwd, float* scale_fwd, void* codes_dgrad,
                        int64_t ld_dgrad, float* scale_dgrad) {
  const int cbytes = code_bytes(code_type(bits, n_groups));
  memset(af, 0, sizeof(*af));
  af->x = w;
  af->R = rows;
  af->C = cols;
  af->ld = ld;
  af->Q = q_of_bits(bits);
  af->G = n_groups;
  *ad = *af;
  af->rt = range_out_ch;
  af->codes_t = codes_fwd;
  af->ldt = ld_fwd;
  af->scale_out = scale_fwd;
  set_alignment(af, cbytes);
  ad->rt = range_in_ch;
  ad->codes = codes_dgrad;
  ad->ldc = ld_dgrad;
  ad->scale_out = scale_dgrad;
  set_alignment(ad, cbytes);
}

// ------------------------------------------------------------- a layer's passes
int check_layer_quant(const sq_layer_step* L) {
  const int64_t M = L->M, K = L->K, N = L->N;
  if (K >= (int64_t(1) << 36) || N >= (int64_t(1) << 36)) return fail(SQ_EINVAL, "calibrate: too many columns");
  const struct { int64_t cols, ld, ldt; const void* t; } t[2] = {{K, L->ld_x, L->ld_xt, L->xt_codes},
                                                                {N, L->ld_g, L->ld_gt, L->gt_codes}};
  for (int i = 0; i < 2; ++i) {
    if (t[i].ld < t[i].cols) return fail(SQ_EINVAL, "quantize: ld_codes < cols");
    if (t[i].t != nullptr && t[i].ldt < M) return fail(SQ_EINVAL, "quantize: ld_t < rows");
    if (!quant_grid_ok(M, t[i].cols))
      return fail(SQ_EUNSUPPORTED, "quantize: tensor too large for one launch (%lld x %lld)",
                  static_cast<long long>(M), static_cast<long long>(t[i].cols));
  }
  if (L->ld_wf < K) return fail(SQ_EINVAL, "quantize_weight: ld_fwd < rows");
  if (L->ld_wd < N) return fail(SQ_EINVAL, "quantize_weight: ld_dgrad < cols");
  if (!quant_grid_ok(K, N))
    return fail(SQ_EUNSUPPORTED, "quantize_weight: tensor too large for one launch (%lld x %lld)",
                static_cast<long long>(K), static_cast<long long>(N));
  return SQ_OK;
}

// blocks of a range pass of v in tiles of 4 << lg columns, and across the columns
static int64_t range_blocks(const RangeView& v, int lg, unsigned* gx) {
  const int64_t tc = int64_t(4) << lg, rows = 8 * (256 >> lg);
  const int64_t nx = (v.C + tc - 1) / tc;
  *gx = static_cast<unsigned>(nx);
  return nx * ((v.R + rows - 1) / rows);
}

bool layer_quant_fits(const sq_layer_step* L) {
  // every block index in 31 bits, with room to spare
  const double m = L->M / 32.0 + 1, k = L->K / 32.0 + 1, n = L->N / 32.0 + 1;
  return m * (k + n) + k * n < 1e9;
}

// The codes of a layer's tensors: one launch while its blocks stay within two resident waves
// (four blocks on each SM), where launches and their tails are what counts; above, one launch per
// tensor, each running beside the tail of the one before it, each body with the instruction cache
// and the registers to itself.  Whole steps when the line was drawn, one launch against three:
// 256 x 512 x 512 (4-bit) 24.7 / 26.6 us; 12608 x 768 x 3072 (6-bit) 271 / 261 us,
// 4096 x 11008 x 4096 (8-bit) 957 / 939 us (with the three one after another 123 us where
// beside one another take 115 us: 12544 x 2304 x 256, 4-bit).
constexpr int kLayerQuantWaveBlocks = 8;   // an SM's, in two waves

template <typename CodeT>
static cudaError_t launch_layer_quantize(const LayerQuant& q, unsigned blocks, int sms, cudaStream_t s) {
  if (blocks > static_cast<unsigned>(kLayerQuantWaveBlocks * sms)) {
    QuantArgs g = q.g, wf = q.wf;
    g.beside = wf.beside = 1;
    launch_quantize<CodeT>(q.x, SQ_GRAN_SHIFT, SQ_ROUND_NEAREST_EVEN, quant_grid(q.x), s);
    launch_quantize_weight<CodeT>(wf, q.wd, quant_grid(wf), s);
    launch_quantize<CodeT>(g, SQ_GRAN_SHIFT, SQ_ROUND_STOCHASTIC, quant_grid(g), s);
    return cudaGetLastError();
  }
  const bool aligned = q.x.form == kAligned && q.g.form == kAligned && q.wf.form == kAligned;
  return aligned ? launch_pdl(layer_quantize_kernel<CodeT, kAligned>, dim3(blocks), dim3(kQuantThreads), s, q)
                 : launch_pdl(layer_quantize_kernel<CodeT, kShifted>, dim3(blocks), dim3(kQuantThreads), s, q);
}

int quantize_layer(const sq_layer_step* L, uint64_t seed, unsigned* words, const ZeroRegion* zero, int nzero,
                   cudaStream_t s) {
  const int64_t M = L->M, K = L->K, N = L->N;
  const int cbytes = code_bytes(code_type(L->bits, L->n_groups));
  const int sms = device_sms(nullptr);
  if (sms <= 0) return fail(SQ_ECUDA, "layer_step: no current CUDA device");
  unsigned* xtau = words + kTauSlots;
  unsigned* gtau = words + 2 * kTauSlots;
  auto bits = [](float* p) { return reinterpret_cast<unsigned*>(p); };
  // 1. accumulators
  LayerInit z = {{bits(L->x_range), bits(L->g_range), bits(L->wf_range), bits(L->wd_range), words},
                 {K, N, N, K, 3 * kTauSlots}};
  const int64_t widest = K > N ? K : N;
  const int64_t ib = (widest + 255) / 256;
  cudaError_t err = launch_pdl(layer_init_kernel, dim3(static_cast<unsigned>(ib < sms ? ib : sms)), dim3(256), s, z);
  if (err != cudaSuccess) return cuda_fail(err, "layer_init_kernel launch");
  // 2. ranges
  LayerRange r;
  memset(&r, 0, sizeof(r));
  r.w = range_view(L->w, K, N, N, false);
  r.g = range_view(L->dy, M, N, N, true);
  r.x = range_view(L->x, M, K, K, true);
  r.glg = range_lg(r.g.C);
  r.xlg = range_lg(r.x.C);
  // runs of column blocks only where a weight is wide (see weight_range_kernel)
  r.wrun = N > kRangeClusterMaxCols ? kWeightRun : 1;
  int64_t blocks = 0;
  for (int k = 0; k < nzero; ++k) {
    r.zero[k] = static_cast<uint4*>(zero[k].p);
    r.zvecs[k] = static_cast<int64_t>(zero[k].bytes / 16);
    r.zblocks[k] = static_cast<unsigned>((r.zvecs[k] + kZeroVecs - 1) / kZeroVecs);
    blocks += r.zblocks[k];
  }
  r.zend = static_cast<unsigned>(blocks);
  r.wgx = static_cast<unsigned>(((N + 127) / 128 + r.wrun - 1) / r.wrun);
  blocks += r.wgx * ((K + 63) / 64);
  r.wend = static_cast<unsigned>(blocks);
  blocks += range_blocks(r.g, r.glg, &r.ggx);
  r.gend = static_cast<unsigned>(blocks);
  blocks += range_blocks(r.x, r.xlg, &r.xgx);
  r.wcols = bits(L->wf_range);
  r.wrows = bits(L->wd_range);
  r.gcols = bits(L->g_range);
  r.xcols = bits(L->x_range);
  r.gtau = gtau;
  r.xtau = xtau;
  r.status = L->dev_status;
  const bool plain = r.x.form == kViewVec && r.g.form == kViewVec && r.w.form == kViewVec;
  err = launch_pdl(plain ? layer_range_kernel<true> : layer_range_kernel<false>, dim3(static_cast<unsigned>(blocks)),
                   dim3(256), s, r);
  if (err != cudaSuccess) return cuda_fail(err, "layer_range_kernel launch");
  // 3. codes
  LayerQuant q;
  memset(&q, 0, sizeof(q));
  auto tensor = [&](QuantArgs* a, const float* x, int64_t cols, const float* range, unsigned* tau, float* tau0,
                    uint8_t* exp, void* codes, int64_t ldc, void* codes_t, int64_t ldt, float* scale) {
    a->x = x;
    a->R = M;
    a->C = a->ld = cols;
    a->Q = q_of_bits(L->bits);
    a->G = L->n_groups;
    a->tslots = tau;
    a->tau_out = tau0;
    a->crange = range;
    a->exp_out = exp;
    a->codes = codes;
    a->ldc = ldc;
    a->codes_t = codes_t;
    a->ldt = ldt;
    a->scale_out = scale;
    set_alignment(a, cbytes);
  };
  tensor(&q.x, L->x, K, L->x_range, xtau, L->x_tau0, L->x_exp, L->x_codes, L->ld_x, L->xt_codes, L->ld_xt, L->x_scale);
  tensor(&q.g, L->dy, N, L->g_range, gtau, L->g_tau0, L->g_exp, L->g_codes, L->ld_g, L->gt_codes, L->ld_gt, L->g_scale);
  q.g.seed = seed;
  weight_args(&q.wf, &q.wd, L->w, K, N, N, L->bits, L->n_groups, L->wf_range, L->wd_range, L->wf_codes, L->ld_wf,
              L->wf_scale, L->wd_codes, L->ld_wd, L->wd_scale);
  q.wf.frange = L->x_range;   // the forward role's rows are X's channels
  q.wf.ftslots = xtau;
  q.wd.frange = L->g_range;   // the loss-propagation role's columns are dY's
  q.wd.ftslots = gtau;
  const dim3 xg = quant_grid(q.x), gg = quant_grid(q.g), wg = quant_grid(q.wf);
  q.xgx = xg.x;
  q.ggx = gg.x;
  q.wgx = wg.x;
  q.xend = xg.x * xg.y;
  q.wend = q.xend + wg.x * wg.y;
  const unsigned nb = q.wend + gg.x * gg.y;
  err = code_type(L->bits, L->n_groups) == SQ_CODE_E4M3 ? launch_layer_quantize<uint8_t>(q, nb, sms, s)
                                                        : launch_layer_quantize<uint16_t>(q, nb, sms, s);
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "layer_quantize_kernel launch");
}

}  // namespace sq

using namespace sq;

// ===================================================================== C entry points
extern "C" int shiftquant_code_type(int bits, int n_groups) {
  if (!bits_ok(bits) || !groups_ok(n_groups))
    return fail(SQ_EINVAL, "bits must be in [2, 8] and n_groups in [1, 8] (got %d, %d)", bits,
                n_groups);
  return code_type(bits, n_groups);
}

extern "C" int shiftquant_code_bytes(int bits, int n_groups) {
  const int t = shiftquant_code_type(bits, n_groups);
  return t < 0 ? t : code_bytes(t);
}

extern "C" const char* shiftquant_status_string(sq_status s) {
  switch (s) {
    case SQ_OK: return "ok";
    case SQ_EINVAL: return "invalid argument";
    case SQ_EALIGN: return "alignment";
    case SQ_EUNSUPPORTED: return "unsupported combination";
    case SQ_ECUDA: return "CUDA error";
    default: return "unknown status";
  }
}

extern "C" const char* shiftquant_last_error(void) { return g_last_error; }

extern "C" sq_status shiftquant_calibrate(const float* x, int64_t rows, int64_t cols,
                                          int64_t ld, int gran, int n_groups,
                                          float* range_out, float* tau0_out, uint8_t* exp_out,
                                          int32_t* dev_status, void* stream) {
  clear_error();
  if (rows < 0 || cols < 0) return fail(SQ_EINVAL, "calibrate: negative size");
  if (cols >= (int64_t(1) << 36)) return fail(SQ_EINVAL, "calibrate: too many columns");
  if (gran < SQ_GRAN_SHIFT || gran > SQ_GRAN_PER_ROW) return fail(SQ_EINVAL, "calibrate: bad gran %d", gran);
  if (gran == SQ_GRAN_SHIFT && !groups_ok(n_groups))
    return fail(SQ_EINVAL, "calibrate: n_groups must be in [1, 8]");
  if (rows > 0 && cols > 0 && (x == nullptr || ld < cols))
    return fail(SQ_EINVAL, "calibrate: x is NULL or ld < cols");
  const int64_t channels = gran == SQ_GRAN_PER_ROW ? rows : cols;
  if (dev_status == nullptr || (channels > 0 && range_out == nullptr))
    return fail(SQ_EINVAL, "calibrate: range_out and dev_status are required");
  if (gran == SQ_GRAN_SHIFT && (tau0_out == nullptr || (cols > 0 && exp_out == nullptr)))
    return fail(SQ_EINVAL, "calibrate: SHIFT needs tau0_out and exp_out");
  cudaStream_t s = as_stream(stream);
  cudaError_t err;
  if (gran == SQ_GRAN_PER_ROW) {
    if (rows == 0) return SQ_OK;
    if (cols == 0) {
      err = cudaMemsetAsync(range_out, 0, sizeof(float) * rows, s);
      return err == cudaSuccess ? SQ_OK : cuda_fail(err, "cudaMemsetAsync");
    }
    const int vec = (ld % 4 == 0) && aligned16(x);
    const int per_block = 8;
    const int64_t blocks = (rows + per_block - 1) / per_block;
    rowmax_kernel<<<static_cast<unsigned>(blocks), per_block * 32, 0, s>>>(x, rows, cols, ld, vec,
                                                                           range_out, dev_status);
    err = cudaGetLastError();
    return err == cudaSuccess ? SQ_OK : cuda_fail(err, "rowmax_kernel launch");
  }
  const bool shift = gran == SQ_GRAN_SHIFT;
  if (rows == 0 || cols == 0) {
    // every range is 0: tau_0 = 0 and every channel in the last group
    if (cols > 0) {
      err = cudaMemsetAsync(range_out, 0, sizeof(float) * cols, s);
      if (err == cudaSuccess && shift) err = cudaMemsetAsync(exp_out, n_groups - 1, cols, s);
      if (err != cudaSuccess) return cuda_fail(err, "cudaMemsetAsync");
    }
    if (shift) {
      err = cudaMemsetAsync(tau0_out, 0, sizeof(float), s);
      if (err != cudaSuccess) return cuda_fail(err, "cudaMemsetAsync");
    }
    return SQ_OK;
  }
  {
    const int64_t iblocks = (cols + 255) / 256;
    calib_init_kernel<<<static_cast<unsigned>(iblocks < 1024 ? iblocks : 1024), 256, 0, s>>>(
        reinterpret_cast<unsigned*>(range_out), cols, nullptr, 0);
    err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "calib_init_kernel launch");
  }
  unsigned* bits = reinterpret_cast<unsigned*>(range_out);
  err = launch_range(x, rows, cols, ld, bits, nullptr, dev_status, s);
  if (err != cudaSuccess) return cuda_fail(err, "colmax_kernel launch");
  if (!shift) return SQ_OK;
  // grouping (Eq. 3) by one block behind the range pass
  err = cols <= static_cast<int64_t>(kGroupSmallThreads) * kGroupPerThread
            ? launch_pdl(group_kernel<kGroupSmallThreads>, dim3(1), dim3(kGroupSmallThreads), s,
                         static_cast<const unsigned*>(bits), cols, n_groups, tau0_out, exp_out, dev_status)
            : launch_pdl(group_kernel<kGroupLargeThreads>, dim3(1), dim3(kGroupLargeThreads), s,
                         static_cast<const unsigned*>(bits), cols, n_groups, tau0_out, exp_out, dev_status);
  if (err == cudaSuccess) err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "group_kernel launch");
}

extern "C" sq_status shiftquant_group(const float* range, int64_t channels, int n_groups,
                                      float* tau0_out, uint8_t* exp_out, int32_t* dev_status,
                                      void* stream) {
  clear_error();
  if (!groups_ok(n_groups)) return fail(SQ_EINVAL, "group: n_groups must be in [1, 8]");
  if (channels < 0) return fail(SQ_EINVAL, "group: negative size");
  if (tau0_out == nullptr || dev_status == nullptr || (channels > 0 && (range == nullptr || exp_out == nullptr)))
    return fail(SQ_EINVAL, "group: range, tau0_out, exp_out and dev_status are required");
  cudaStream_t s = as_stream(stream);
  if (channels == 0) {
    const cudaError_t err = cudaMemsetAsync(tau0_out, 0, sizeof(float), s);
    return err == cudaSuccess ? SQ_OK : cuda_fail(err, "cudaMemsetAsync");
  }
  const unsigned* rb = reinterpret_cast<const unsigned*>(range);
  if (channels <= static_cast<int64_t>(kGroupSmallThreads) * kGroupPerThread)
    group_kernel<kGroupSmallThreads><<<1, kGroupSmallThreads, 0, s>>>(rb, channels, n_groups, tau0_out,
                                                                     exp_out, dev_status);
  else
    group_kernel<kGroupLargeThreads><<<1, kGroupLargeThreads, 0, s>>>(rb, channels, n_groups, tau0_out,
                                                                     exp_out, dev_status);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "group_kernel launch");
}

extern "C" sq_status shiftquant_quantize(const float* x, int64_t rows, int64_t cols, int64_t ld,
                                         int gran, int bits, int n_groups,
                                         const float* range_or_tau0, const uint8_t* exp,
                                         const uint8_t* fold_exp, int mode, uint64_t seed,
                                         int64_t row0, void* codes, int64_t ld_codes,
                                         void* codes_t, int64_t ld_t, float* scale_out,
                                         void* stream) {
  clear_error();
  if (!bits_ok(bits) || !groups_ok(n_groups))
    return fail(SQ_EINVAL, "quantize: bits must be in [2, 8] and n_groups in [1, 8]");
  if (rows < 0 || cols < 0) return fail(SQ_EINVAL, "quantize: negative size");
  if (row0 < 0) return fail(SQ_EINVAL, "quantize: negative row0");
  if (gran < SQ_GRAN_SHIFT || gran > SQ_GRAN_PER_ROW) return fail(SQ_EINVAL, "quantize: bad gran");
  if (mode != SQ_ROUND_NEAREST_EVEN && mode != SQ_ROUND_STOCHASTIC)
    return fail(SQ_EINVAL, "quantize: bad rounding mode");
  if (gran == SQ_GRAN_SHIFT && fold_exp != nullptr)
    return fail(SQ_EINVAL, "quantize: SHIFT takes no fold_exp");
  cudaStream_t s = as_stream(stream);
  const int type = code_type(bits, n_groups);
  const int cbytes = code_bytes(type);
  if (rows == 0 || cols == 0) {
    // every range is 0: scales are 0 and there is no code to write
    const int64_t n = gran == SQ_GRAN_SHIFT ? 1 : (gran == SQ_GRAN_PER_COL ? cols : rows);
    if (n == 0) return SQ_OK;
    if (scale_out == nullptr) return fail(SQ_EINVAL, "quantize: scale_out is required");
    cudaError_t err = cudaMemsetAsync(scale_out, 0, sizeof(float) * n, s);
    return err == cudaSuccess ? SQ_OK : cuda_fail(err, "cudaMemsetAsync");
  }
  if (range_or_tau0 == nullptr || scale_out == nullptr)
    return fail(SQ_EINVAL, "quantize: range_or_tau0 and scale_out are required");
  if (gran == SQ_GRAN_SHIFT && exp == nullptr)
    return fail(SQ_EINVAL, "quantize: SHIFT needs exp");
  if (codes == nullptr && codes_t == nullptr)
    return fail(SQ_EINVAL, "quantize: at least one of codes / codes_t is required");
  if (codes && ld_codes < cols) return fail(SQ_EINVAL, "quantize: ld_codes < cols");
  if (codes_t && ld_t < rows) return fail(SQ_EINVAL, "quantize: ld_t < rows");
  if (x == nullptr || ld < cols) return fail(SQ_EINVAL, "quantize: x is NULL or ld < cols");
  QuantArgs a;
  memset(&a, 0, sizeof(a));
  a.x = x;
  a.R = rows;
  a.C = cols;
  a.ld = ld;
  a.Q = q_of_bits(bits);
  a.G = n_groups;
  a.seed = seed;
  a.row0 = row0;
  a.rt = range_or_tau0;
  a.exp = exp;
  a.fold = fold_exp;
  a.codes = codes;
  a.ldc = ld_codes;
  a.codes_t = codes_t;
  a.ldt = ld_t;
  a.scale_out = scale_out;
  a.pos_cols = g_order_cols;
  a.pos_rows = g_order_rows;
  set_alignment(&a, cbytes);
  if (!quant_grid_ok(rows, cols))
    return fail(SQ_EUNSUPPORTED, "quantize: tensor too large for one launch (%lld x %lld)",
                static_cast<long long>(rows), static_cast<long long>(cols));
  const dim3 grid = quant_grid(a);
  if (type == SQ_CODE_E4M3)
    launch_quantize<uint8_t>(a, gran, mode, grid, s);
  else
    launch_quantize<uint16_t>(a, gran, mode, grid, s);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "quantize_kernel launch");
}

// ------------------------------------------------------------------ group order
extern "C" int64_t shiftquant_group_order_width(int64_t channels, int bits, int n_groups) {
  if (channels < 0 || !bits_ok(bits) || !groups_ok(n_groups)) return -1;
  const int64_t bk = 128 / code_bytes(code_type(bits, n_groups));
  return (channels + bk - 1) / bk * bk + (n_groups - 1) * bk;
}

extern "C" sq_status shiftquant_group_order(const uint8_t* exp, int64_t channels, int bits,
                                            int n_groups, int32_t* pos_out, int32_t* seg_out,
                                            void* stream) {
  clear_error();
  if (!bits_ok(bits) || !groups_ok(n_groups))
    return fail(SQ_EINVAL, "group_order: bits must be in [2, 8] and n_groups in [1, 8]");
  if (channels < 0 || channels > INT32_MAX / 2) return fail(SQ_EINVAL, "group_order: bad channel count");
  if (seg_out == nullptr || (channels > 0 && (exp == nullptr || pos_out == nullptr)))
    return fail(SQ_EINVAL, "group_order: exp, pos_out and seg_out are required");
  const int bk = 128 / code_bytes(code_type(bits, n_groups));
  group_order_kernel<<<1, kOrderThreads, 0, as_stream(stream)>>>(exp, channels, n_groups, bk,
                                                                   pos_out, seg_out);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "group_order_kernel launch");
}

extern "C" sq_status shiftquant_quantize_ordered(const float* x, int64_t rows, int64_t cols,
                                                 int64_t ld, int gran, int bits, int n_groups,
                                                 const float* range_or_tau0, const uint8_t* exp,
                                                 int mode, uint64_t seed, int64_t row0,
                                                 const int32_t* pos, const int32_t* seg,
                                                 void* codes, int64_t ld_codes, void* codes_t,
                                                 int64_t ld_t, float* scale_out, void* stream) {
  clear_error();
  if (pos == nullptr || seg == nullptr) return fail(SQ_EINVAL, "quantize_ordered: pos and seg are required");
  if (!bits_ok(bits) || !groups_ok(n_groups))
    return fail(SQ_EINVAL, "quantize_ordered: bits must be in [2, 8] and n_groups in [1, 8]");
  // the ordered output: codes for ShiftQuant and per-row grans, codes_t for per-column
  const bool on_t = gran == SQ_GRAN_PER_COL;
  void* ordered = on_t ? codes_t : codes;
  const int64_t ord_rows = on_t ? cols : rows;       // rows of the ordered buffer
  const int64_t ord_ld = on_t ? ld_t : ld_codes;
  const int64_t chans = on_t ? rows : cols;          // the ordered (inner) index
  if (ordered == nullptr)
    return fail(SQ_EINVAL, "quantize_ordered: the group-ordered output (%s) is required",
                on_t ? "codes_t" : "codes");
  const int64_t width = shiftquant_group_order_width(chans, bits, n_groups);
  if (ord_ld < width)
    return fail(SQ_EINVAL, "quantize_ordered: the ordered output needs a leading dimension of "
                "at least %lld (shiftquant_group_order_width)", static_cast<long long>(width));
  // the other output (if any) keeps the natural order; a leading dimension >= the natural
  // width is checked by the plain quantizer below
  g_order_cols = on_t ? nullptr : pos;
  g_order_rows = on_t ? pos : nullptr;
  const sq_status st = shiftquant_quantize(x, rows, cols, ld, gran, bits, n_groups, range_or_tau0,
                                           exp, nullptr, mode, seed, row0, codes, ld_codes, codes_t,
                                           ld_t, scale_out, stream);
  g_order_cols = g_order_rows = nullptr;
  if (st != SQ_OK || ord_rows == 0) return st;
  cudaStream_t s = as_stream(stream);
  int64_t blocks = (ord_rows + 7) / 8;
  if (blocks > 4096) blocks = 4096;
  if (code_type(bits, n_groups) == SQ_CODE_E4M3)
    order_pad_kernel<uint8_t><<<static_cast<unsigned>(blocks), 256, 0, s>>>(
        static_cast<uint8_t*>(ordered), ord_rows, ord_ld, seg, n_groups);
  else
    order_pad_kernel<uint16_t><<<static_cast<unsigned>(blocks), 256, 0, s>>>(
        static_cast<uint16_t*>(ordered), ord_rows, ord_ld, seg, n_groups);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "order_pad_kernel launch");
}

extern "C" sq_status shiftquant_calibrate_weight(const float* w, int64_t rows, int64_t cols,
                                                 int64_t ld, float* range_out_ch,
                                                 float* range_in_ch, int32_t* dev_status,
                                                 void* stream) {
  clear_error();
  if (rows < 0 || cols < 0) return fail(SQ_EINVAL, "calibrate_weight: negative size");
  if (cols >= (int64_t(1) << 36)) return fail(SQ_EINVAL, "calibrate_weight: too many columns");
  if (rows > 0 && cols > 0 && (w == nullptr || ld < cols))
    return fail(SQ_EINVAL, "calibrate_weight: w is NULL or ld < cols");
  if (dev_status == nullptr || (cols > 0 && range_out_ch == nullptr) ||
      (rows > 0 && range_in_ch == nullptr))
    return fail(SQ_EINVAL, "calibrate_weight: range_out_ch, range_in_ch and dev_status are required");
  cudaStream_t s = as_stream(stream);
  cudaError_t err;
  if (rows == 0 || cols == 0) {
    // every range is 0
    if (cols > 0 && (err = cudaMemsetAsync(range_out_ch, 0, sizeof(float) * cols, s)) != cudaSuccess)
      return cuda_fail(err, "cudaMemsetAsync");
    if (rows > 0 && (err = cudaMemsetAsync(range_in_ch, 0, sizeof(float) * rows, s)) != cudaSuccess)
      return cuda_fail(err, "cudaMemsetAsync");
    return SQ_OK;
  }
  unsigned* cb = reinterpret_cast<unsigned*>(range_out_ch);
  unsigned* rb = reinterpret_cast<unsigned*>(range_in_ch);
  // Both ranges from one read.  On wide weights the blocks of one row tile run together and
  // their per-row atomics (one per 128 columns) partly serialise; measured on a
  // [4096, 11008] weight this pass (58 us) still beats a column pass plus a one-warp-per-row
  // pass (34 + 30 us).
  const int64_t n = rows > cols ? rows : cols;
  const int64_t iblocks = (n + 255) / 256;
  calib_init_kernel<<<static_cast<unsigned>(iblocks < 1024 ? iblocks : 1024), 256, 0, s>>>(
      cb, cols, rb, rows);
  err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, "calib_init_kernel launch");
  err = launch_range(w, rows, cols, ld, cb, rb, dev_status, s);
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "colmax_kernel launch");
}

extern "C" sq_status shiftquant_quantize_weight(const float* w, int64_t rows, int64_t cols,
                                                int64_t ld, int bits, int n_groups,
                                                const float* range_out_ch, const float* range_in_ch,
                                                const uint8_t* fold_fwd, const uint8_t* fold_dgrad,
                                                void* codes_fwd, int64_t ld_fwd, float* scale_fwd,
                                                void* codes_dgrad, int64_t ld_dgrad,
                                                float* scale_dgrad, void* stream) {
  clear_error();
  if (!bits_ok(bits) || !groups_ok(n_groups))
    return fail(SQ_EINVAL, "quantize_weight: bits must be in [2, 8] and n_groups in [1, 8]");
  if (rows < 0 || cols < 0) return fail(SQ_EINVAL, "quantize_weight: negative size");
  cudaStream_t s = as_stream(stream);
  const int type = code_type(bits, n_groups);
  const int cbytes = code_bytes(type);
  if (rows == 0 || cols == 0) {
    // every range is 0: the scales are 0 and there is no code to write
    cudaError_t err;
    if (cols > 0) {
      if (scale_fwd == nullptr) return fail(SQ_EINVAL, "quantize_weight: scale_fwd is required");
      if ((err = cudaMemsetAsync(scale_fwd, 0, sizeof(float) * cols, s)) != cudaSuccess)
        return cuda_fail(err, "cudaMemsetAsync");
    }
    if (rows > 0) {
      if (scale_dgrad == nullptr) return fail(SQ_EINVAL, "quantize_weight: scale_dgrad is required");
      if ((err = cudaMemsetAsync(scale_dgrad, 0, sizeof(float) * rows, s)) != cudaSuccess)
        return cuda_fail(err, "cudaMemsetAsync");
    }
    return SQ_OK;
  }
  if (w == nullptr || ld < cols) return fail(SQ_EINVAL, "quantize_weight: w is NULL or ld < cols");
  if (range_out_ch == nullptr || range_in_ch == nullptr || scale_fwd == nullptr ||
      scale_dgrad == nullptr || codes_fwd == nullptr || codes_dgrad == nullptr)
    return fail(SQ_EINVAL, "quantize_weight: ranges, codes and scales of both roles are required");
  if (ld_fwd < rows) return fail(SQ_EINVAL, "quantize_weight: ld_fwd < rows");
  if (ld_dgrad < cols) return fail(SQ_EINVAL, "quantize_weight: ld_dgrad < cols");
  QuantArgs af, ad;
  weight_args(&af, &ad, w, rows, cols, ld, bits, n_groups, range_out_ch, range_in_ch, codes_fwd, ld_fwd,
              scale_fwd, codes_dgrad, ld_dgrad, scale_dgrad);
  af.fold = fold_fwd;
  ad.fold = fold_dgrad;
  if (!quant_grid_ok(rows, cols))
    return fail(SQ_EUNSUPPORTED, "quantize_weight: tensor too large for one launch (%lld x %lld)",
                static_cast<long long>(rows), static_cast<long long>(cols));
  const dim3 grid = quant_grid(af);
  if (type == SQ_CODE_E4M3)
    launch_quantize_weight<uint8_t>(af, ad, grid, s);
  else
    launch_quantize_weight<uint16_t>(af, ad, grid, s);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? SQ_OK : cuda_fail(err, "quantize_weight_kernel launch");
}
