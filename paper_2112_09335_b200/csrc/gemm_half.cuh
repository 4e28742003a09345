// Dense product C[M x N] = A[M x K] * B with operands split into pairs of halves, on the 5th-generation tensor cores: the form
// of the feature-by-weight contractions on graphs of thousands of rows (k_gemm_tc_ws, TF32 pairs, has the rest).
//
// fp32 accuracy from fp16 hardware: a row of A is scaled by a power of two that brings its largest element into [2^14, 2^15)
// (exact), so is a column of B (or all of B by a bound of its elements), and each scaled element x is split into x_hi = half(x) and x_lo = half(2^11 (x - x_hi)).  Both
// hold 11 bits and are rounded to nearest, so x_hi + 2^-11 x_lo is x to 2^-23 of its magnitude where that is 2^-13 or more, that is for
// elements down to 2^-27 of the largest of their row; below, bits of x_lo fall under the smallest half and the element is held to
// 2^-50 of that largest one only.  Where that could show, rows are formed by TF32 pairs instead (redo_rows): all of them where B holds
// such an element (its image says); where B is wide, those whose row of A does (the producers look).  B is wide where an element,
// zero included, is below 2^-8 (the largest is 2^14 or more).  Beside a B that is not, K elements held to 2^-36 (2^15 is the largest)
// cost at most K 2^-36 2^15 against sum |a||b| >= 2^14 2^-8: K 2^-27, and with the accumulator's (K / 16 + 3.5) 2^-23 that
// is within the bound of TF32 pairs, (K / 8 + 11) 2^-23.  As with TF32 pairs,
//   A B ~= A_hi B_hi + 2^-11 (A_lo B_hi + A_hi B_lo)
// is accumulated in fp32, the main product and the corrections apart (the tensor core rounds an accumulator toward zero at every
// MMA); the scales come off in the epilogue.  Against TF32 pairs an MMA covers twice the reduction in the same time (and the
// accumulator is rounded half as often: errors against fp64 halve, 6.4e-7 -> 3.4e-7 of ||C|| at K = 256), and the operands take
// half the shared memory and half of its bandwidth, which bounded the TF32 form at 256 columns.
//
// 1.2 M rows, launched alone, TF32 pairs -> this form in ms (HBM alone): 256 x 256 0.81 -> 0.59 (0.38), 128 x 256 0.46 -> 0.38 (0.28),
// 256 x 128 0.43 -> 0.36 (0.28), 47 x 256 0.33 -> 0.31 (0.22), 256 x 47 0.31 -> 0.26 (0.22).  At 256 columns shared memory is what is left: a K chunk of 32 moves
// 72 KB of MMA operands, 48 KB of copies, 32 KB of splitting and 48 KB of the epilogue through it, 1,560 clocks at 128 B a clock
// against 768 of MMAs; leaving out the copies of B, the splitting or the stores alone saves 4, 13 and 10 %.  Columns in one group
// of 256 instead of two of 128 (every A tile read and split twice): 0.59 against 0.67 ms.
//
// The row maxima of A come with A: whoever writes the matrix leaves them (row_max).  B comes as an image of the staged layout, kept
// by whoever writes the weights (put_half: every column by one scale, from a bound of the matrix) or made by k_split_b from a finished
// gradient (every column by its own: a bound kept with the partial sums, in the writer itself, is 2^5 to 2^7 above the largest element, and
// with it a 767 x 1000 gradient always held elements too small for a pair; the launch takes 6 to 8 us under a profiler).
#pragma once
#include <cfloat>
#include <cuda_fp16.h>

#include "gemm_tc.cuh"

namespace gtc {

constexpr int kHalfRow = kChunkK * 2;              // 64 bytes: a row of an operand tile, 64-byte swizzle
constexpr int kHalfGroup = 8 * kHalfRow;           // 512 bytes: eight of them
constexpr float kLoScale = 2048.f;

// Byte offset of the 16-byte unit `u` (0..3, eight halves) of row `r` in a K-major operand tile with the 64-byte swizzle.
__device__ __forceinline__ uint32_t swz_half(int r, int u) { return (uint32_t)r * kHalfRow + (uint32_t)((u ^ ((r >> 1) & 3)) << 4); }
// Operand descriptors: version 1, SWIZZLE_64B (low word as for the 128-byte swizzle); 8-row groups of B one after the other, those
// of A_hi and A_lo in turn (see the producers).
constexpr uint32_t kDescHiA = (2 * kHalfGroup >> 4) | (1u << 14) | (4u << 29);
constexpr uint32_t kDescHiB = (kHalfGroup >> 4) | (1u << 14) | (4u << 29);
// Instruction descriptor: D fp32, A and B fp16, both K-major, M = 128, N = nt.
__device__ __forceinline__ uint32_t instr_desc_half(int nt) {
  return (1u << 4) | ((uint32_t)(nt >> 3) << 17) | ((uint32_t)(kBlockM >> 4) << 24);
}
__device__ __forceinline__ void mma_half(uint32_t tmem_d, uint32_t da_lo, uint32_t db_lo, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %6};\n\t"
      "mov.b64 db, {%2, %7};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, {%5, %5, %5, %5}, p;\n\t}"
      ::"r"(tmem_d), "r"(da_lo), "r"(db_lo), "r"(idesc), "r"(accumulate), "r"(0u), "r"(kDescHiA), "r"(kDescHiB)
      : "memory");
}

// The power of two that brings m (the largest magnitude of a row) into [2^14, 2^15), and its inverse.  Both stay normal numbers:
// rows whose largest element is below 2^-111 are scaled by 2^126.  m = 0, an infinity and a NaN give some scale; infinite and NaN
// elements then reach the result as NaN.
__device__ __forceinline__ uint32_t scale_field(float m) { return (uint32_t)min(253, max(1, 268 - (int)(__float_as_uint(m) >> 23))); }
__device__ __forceinline__ float scale_of(float m) { return __uint_as_float(scale_field(m) << 23); }
__device__ __forceinline__ float inverse_scale_of(float m) { return __uint_as_float((254u - scale_field(m)) << 23); }

// Elements too small for a pair.  Keys order magnitudes with zero, which every pair holds, behind all others; below_pairs(scale) is the
// key below which a scaled element lies under 2^-13, marks_for the marks an element of B makes.  Where the largest element is not
// finite (scale 2^-114) there is no such key: the row is NaN in any form.  Under a scale of 2^114 or more (largest element below
// 2^-98) subnormal elements count as too small.
__host__ __device__ __forceinline__ uint32_t size_key(uint32_t bits) { return (bits << 1) - 1u; }
__device__ __forceinline__ uint32_t size_key(float x) { return size_key(__float_as_uint(x)); }
__device__ __forceinline__ uint32_t below_pairs(float scale) {
  const int field = (int)(__float_as_uint(scale) >> 23);
  return field == 13 ? 0u : size_key((uint32_t)max(1, 241 - field) << 23);
}
constexpr int kBelowPairs = 1, kWide = 2;
__device__ __forceinline__ int marks_for(float x, float scale) {
  return (size_key(x) < below_pairs(scale) ? kBelowPairs : 0) | (fabsf(x * scale) < 0x1p-8f ? kWide : 0);
}
__device__ __forceinline__ uint32_t least_key(const float4& a) {
  return min(__vimin3_u32(size_key(a.x), size_key(a.y), size_key(a.z)), size_key(a.w));
}
__device__ __forceinline__ uint32_t least_key(const float4& a, const float4& b) {
  return __vimin3_u32(least_key(a), __vimin3_u32(size_key(b.x), size_key(b.y), size_key(b.z)), size_key(b.w));
}

// Eight scaled elements as halves: hi rounded to nearest, lo = half(2^11 (x - hi)), the difference exact.
__device__ __forceinline__ void split_pair(float x0, float x1, float scale, uint32_t& hi, uint32_t& lo) {
  const float y0 = x0 * scale, y1 = x1 * scale;
  const __half2 h = __floats2half2_rn(y0, y1);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(fmaf(-kLoScale, f.x, kLoScale * y0), fmaf(-kLoScale, f.y, kLoScale * y1));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ void split_unit(const float4& a, const float4& b, float scale, uint4& hi, uint4& lo) {
  split_pair(a.x, a.y, scale, hi.x, lo.x);
  split_pair(a.z, a.w, scale, hi.y, lo.y);
  split_pair(b.x, b.y, scale, hi.z, lo.z);
  split_pair(b.z, b.w, scale, hi.w, lo.w);
}

// The weight operand, split in the layout the MMA descriptors read.  For column group g (nt columns) and K chunk kc: the nt x 32
// tile of B_hi followed by that of B_lo, one contiguous block of 2 * nt * 64 bytes at block index g * kc_count + kc, which a stage
// gets by one bulk copy; behind all blocks the inverse scale of every column, nt per group, and the marks: words that hold kBelowPairs or
// kWide where elements ask for it.  A writer has a word of its own for each column or each 32 x 32 elements it
// writes, the first of them among these; one that marks the whole image (put_marks) sets that first word and clears the others, so that
// whoever writes the image next, by tiles, leaves none of its marks behind.
struct Image {
  uint8_t* data;   // NULL: no image is kept
  int nt, kc;      // column group width, K chunks
};
__host__ __device__ inline size_t image_blocks_bytes(int groups, int nt, int kc) { return (size_t)groups * kc * 2 * nt * kHalfRow; }
__host__ __device__ inline int image_marks(int groups, int nt, int kc) { return max(groups * nt, kc * ((groups * nt + 31) / 32)); }
__device__ __forceinline__ int* marks_of(const Image& im, int n) {
  const int groups = (n + im.nt - 1) / im.nt;
  return reinterpret_cast<int*>(im.data + image_blocks_bytes(groups, im.nt, im.kc)) + groups * im.nt;
}
// The marks of a whole image of `n` columns, by the threads of one block.
__device__ __forceinline__ void put_marks(const Image& im, int n, int marks) {
  if (im.data == nullptr) return;
  int* const at = marks_of(im, n);
  for (int i = threadIdx.x; i < image_marks((n + im.nt - 1) / im.nt, im.nt, im.kc); i += blockDim.x) at[i] = i == 0 ? marks : 0;
}
// One element of an image: B[k][n] = x, already scaled.  The padding of an image is zero from the start and never written.
__device__ __forceinline__ void put_half(const Image& im, int n, int k, float x) {
  if (im.data == nullptr) return;
  const int g = n / im.nt, r = n - g * im.nt, c = k / kChunkK, kk = k - c * kChunkK;
  uint8_t* const at = im.data + (size_t)(g * im.kc + c) * (size_t)(2 * im.nt * kHalfRow) + swz_half(r, kk >> 3) + (kk & 7) * 2;
  const __half h = __float2half_rn(x);
  *reinterpret_cast<__half*>(at) = h;
  *reinterpret_cast<__half*>(at + (size_t)im.nt * kHalfRow) = __float2half_rn(fmaf(-kLoScale, __half2float(h), kLoScale * x));
}
// A bound formed from others may leave the range while every element it bounds is finite: the largest number bounds those too.
// Elements that are not finite stay in their column of the product under any finite scale.
__device__ __forceinline__ float finite_bound(float m) { return fminf(m, FLT_MAX); }
// The inverse scales of an image whose `n` columns share the scale of m, a finite number, by the threads of one block.
__device__ __forceinline__ void put_scales(const Image& im, int n, float m) {
  if (im.data == nullptr) return;
  const int groups = (n + im.nt - 1) / im.nt;
  float* const at = reinterpret_cast<float*>(im.data + image_blocks_bytes(groups, im.nt, im.kc));
  for (int c = threadIdx.x; c < groups * im.nt; c += blockDim.x) at[c] = inverse_scale_of(m);
}

struct SplitB {
  const float* Bk;   // N x K, row-major, columns K .. ldbk - 1 zero
  int ldbk, N, K;
  Image image;
};
// kSplitThreads threads per column of B (row of Bk), those that fill the last group up with zeros included, each column with a scale of its
// own.  Between a gradient and its product, so what counts is the chain: a column is loaded at once and split out of registers
// (a
// warp per column, which loops and loads it a second time, took 8.1 instead of 6.1 us between events at 500 x 128).
constexpr int kSplitThreads = 64, kSplitColumns = 256 / kSplitThreads, kSplitUnits = 2048 / 8 / kSplitThreads;   // K <= 2048
__global__ void __launch_bounds__(256)
k_split_b(const SplitB p, int rows) {
  enter_kernel();
  __shared__ uint32_t s_m[8], s_key[8], s_least[8];
  const int warp = threadIdx.x >> 5, first = warp & ~(kSplitThreads / 32 - 1);   // of the column's warps
  const int n = blockIdx.x * kSplitColumns + threadIdx.x / kSplitThreads, t = threadIdx.x % kSplitThreads, nt = p.image.nt;
  const float* const src = p.Bk + (long long)n * p.ldbk;
  const auto load = [&](int k) { return n < p.N && k < p.K ? *reinterpret_cast<const float4*>(src + k) : make_float4(0.f, 0.f, 0.f, 0.f); };
  float4 a[kSplitUnits], b[kSplitUnits];
#pragma unroll
  for (int i = 0; i < kSplitUnits; ++i) {
    const int k = 8 * (t + i * kSplitThreads);
    a[i] = load(k);
    b[i] = load(k + 4);
  }
  float m = 0.f, least = INFINITY;   // zeros count for the least
  uint32_t key = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < kSplitUnits; ++i) {
    const float x[8] = {a[i].x, a[i].y, a[i].z, a[i].w, b[i].x, b[i].y, b[i].z, b[i].w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      m = fmaxf(m, fabsf(x[e]));
      least = 8 * (t + i * kSplitThreads) + e < p.K ? fminf(least, fabsf(x[e])) : least;
    }
    key = min(key, least_key(a[i], b[i]));
  }
  // magnitudes: their order is that of their bits
  const uint32_t warp_m = __reduce_max_sync(0xffffffffu, __float_as_uint(m)), warp_key = __reduce_min_sync(0xffffffffu, key);
  const uint32_t warp_least = __reduce_min_sync(0xffffffffu, __float_as_uint(least));
  if ((threadIdx.x & 31) == 0) { s_m[warp] = warp_m; s_key[warp] = warp_key; s_least[warp] = warp_least; }
  __syncthreads();
  if (n >= rows) return;
  uint32_t top = s_m[first], low_key = s_key[first], low = s_least[first];
#pragma unroll
  for (int w = 1; w < kSplitThreads / 32; ++w) {
    top = max(top, s_m[first + w]);
    low_key = min(low_key, s_key[first + w]);
    low = min(low, s_least[first + w]);
  }
  m = __uint_as_float(top);
  const float scale = scale_of(m);
  const int g = n / nt, r = n - g * nt;
  uint8_t* const at = p.image.data + image_blocks_bytes(g, nt, p.image.kc);
#pragma unroll
  for (int i = 0; i < kSplitUnits; ++i) {
    const int q = t + i * kSplitThreads;
    if (q >= p.image.kc * 4) break;
    uint4 hi, lo;
    split_unit(a[i], b[i], scale, hi, lo);
    uint8_t* const dst = at + (size_t)(q >> 2) * (2 * nt * kHalfRow) + swz_half(r, q & 3);
    *reinterpret_cast<uint4*>(dst) = hi;
    *reinterpret_cast<uint4*>(dst + (size_t)nt * kHalfRow) = lo;
  }
  if (t == 0) {
    const int groups = (p.N + nt - 1) / nt;
    // a column of zeros, padding among them, takes any: 1 joins with the factor of every row that others join with
    reinterpret_cast<float*>(p.image.data + image_blocks_bytes(groups, nt, p.image.kc))[n] = m > 0.f ? inverse_scale_of(m) : 1.f;
    marks_of(p.image, p.N)[n] = n >= p.N ? 0 : (low_key < below_pairs(scale) ? kBelowPairs : 0) | (__uint_as_float(low) * scale < 0x1p-8f ? kWide : 0);
  }
}

template <int NT>
struct HalfCfg {
  static constexpr int kSets = NT > 128 ? 1 : 2;        // accumulator sets (main + correction each)
  // Eight epilogue warps where the column steps divide by two per quarter: with one set the MMAs of the next tile wait for them (and
  // four producer warps leave them the registers), with two and a short reduction they are what a tile takes longest for (1.2 M rows,
  // 128 columns, four -> eight: 201 -> 152 us at K = 12, 207 -> 159 at 47, 238 -> 212 at 128, 358 -> 358 at 256).
  static constexpr int kProdWarps = NT > 128 ? 4 : 8, kEpiWarps = NT >= 64 && NT != 96 ? 8 : 4;
  static constexpr int kMmaWarp = kProdWarps + kEpiWarps;
  static constexpr int kThreads = (kMmaWarp + 2) * 32;
  static constexpr int kBBytes = 2 * NT * kHalfRow;     // hi and lo of a chunk
  static constexpr int kSlot = kATileBytes + kBBytes;   // a tile of A, raw and then split in place, and the chunk of B's image
  static constexpr int kSlots = NT > 128 ? 4 : NT > 64 ? 5 : 8;
  static constexpr int kAccCols = kSets * 2 * NT;
  static constexpr uint32_t kTmemCols = kAccCols <= 64 ? 64 : kAccCols <= 128 ? 128 : kAccCols <= 256 ? 256 : 512;
  static constexpr size_t kSmem = (size_t)kSlots * kSlot + kEpiWarps * 4096 + NT * sizeof(float) + 1024;
  static constexpr int kRedoStage = 2 * kATileBytes + 2 * NT * kChunkK * 4;   // a chunk of both operands as TF32 pairs
  static_assert(2 * kRedoStage <= kSlots * kSlot && kRedoStage % 1024 == 0, "two of them lie where the slots were");
};

// Row tiles of this block whose rows may hold elements too small for a pair: bit i for its i-th tile, the last bit for all from there on.
constexpr int kRedoBits = 2048;

// Rows with elements too small for a pair, or all rows (`all`), of this block's tiles once more, by TF32 pairs: each element has an
// exponent of its own there.  By all threads of the block, after its pipeline has come to rest; shared memory and tensor memory are the
// pipeline's.  Which rows are stored is decided by the rows themselves, so a row's value does not depend on the others of its tile.
// Ordinary data rarely comes here, so this is two stages between barriers and not a pipeline of its own.  us, nothing to redo / one row in
// 100 k / every row: 256 x 256 on 169 k rows 91 / 114 / 341, on 1.2 M 603 / 646 / 2298, 256 x 47 on 1.2 M 271 / 308 / 1079 (all rows by
// k_gemm_tc_ws's pipeline: 0.81 ms, 0.31).  False: a wait ran out.
template <int NT>
__device__ __noinline__ bool redo_rows(const float* __restrict__ A, int lda, const float* __restrict__ row_max, const float* __restrict__ Bk, int ldbk,
                                       float* __restrict__ C, int ldc, int M, int N, int K, const uint32_t* marked, bool all, uint8_t* smem, uint32_t tmem_base,
                                       uint32_t bars, volatile int* abortp) {
  using Cfg = HalfCfg<NT>;
  constexpr int kRows = Cfg::kThreads / 8;   // rows a turn of the block's threads covers, eight 16-byte units each
  constexpr int kPassesA = (kBlockM + kRows - 1) / kRows, kPassesB = (NT + kRows - 1) / kRows;
  constexpr uint32_t kBTile = NT * kChunkK * 4;
  int* const row_marks = reinterpret_cast<int*>(smem + (size_t)Cfg::kSlots * Cfg::kSlot);   // of the tile's rows, where the epilogue's buffers were
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, unit = tid & 7;
  const int n_tiles = (M + kBlockM - 1) / kBlockM, kc_count = (K + kChunkK - 1) / kChunkK, n0 = blockIdx.y * NT;
  int chunk = 0;                             // chunks staged so far: stage chunk & 1, whose commits complete its barrier in turn
  for (int tile = blockIdx.x, tile_i = 0; tile < n_tiles; tile += gridDim.x, ++tile_i) {
    const int bit = min(tile_i, kRedoBits - 1);
    if (!all && !(marked[bit >> 5] >> (bit & 31) & 1u)) continue;
    const long long row0 = (long long)tile * kBlockM;
    if (tid < kBlockM) row_marks[tid] = all;
    float4 va[kPassesA], vb[kPassesB];   // the next chunk's elements, on their way while the one before it is multiplied
    const auto load = [&](int kc) {
      const int k = kc * kChunkK + unit * 4;
      const auto at = [&](const float* p, bool in) { return in && k < K ? *reinterpret_cast<const float4*>(p + k) : make_float4(0.f, 0.f, 0.f, 0.f); };
#pragma unroll
      for (int i = 0; i < kPassesA; ++i) {
        const int r = (tid >> 3) + i * kRows;
        va[i] = at(A + (row0 + r) * lda, r < kBlockM && row0 + r < M);
      }
#pragma unroll
      for (int i = 0; i < kPassesB; ++i) {
        const int r = (tid >> 3) + i * kRows;
        vb[i] = at(Bk + (long long)(n0 + r) * ldbk, r < NT && n0 + r < N);
      }
    };
    load(0);
    for (int kc = 0; kc < kc_count; ++kc, ++chunk) {
      const int stage = chunk & 1;
      const bool ok = chunk < 2 || mbar_wait_abortable(bars + 8 * stage, (uint32_t)((chunk >> 1) - 1) & 1u, abortp);
      if (!__syncthreads_and(ok)) return false;   // and the row marks are set
      uint8_t* const st = smem + (size_t)stage * Cfg::kRedoStage;
      const auto put = [&](uint8_t* at, uint32_t lo_at, const float4& v) {
        float4 h, l;
        split_tf32(v.x, h.x, l.x); split_tf32(v.y, h.y, l.y); split_tf32(v.z, h.z, l.z); split_tf32(v.w, h.w, l.w);
        *reinterpret_cast<float4*>(at) = h;
        *reinterpret_cast<float4*>(at + lo_at) = l;
      };
#pragma unroll
      for (int i = 0; i < kPassesA; ++i) {
        const int r = (tid >> 3) + i * kRows;
        if (r >= kBlockM) break;
        if (row0 + r < M && least_key(va[i]) < below_pairs(scale_of(__ldg(row_max + row0 + r)))) row_marks[r] = 1;
        put(st + swz(r, unit), kATileBytes, va[i]);
      }
#pragma unroll
      for (int i = 0; i < kPassesB; ++i) {
        const int r = (tid >> 3) + i * kRows;
        if (r < NT) put(st + 2 * kATileBytes + swz(r, unit), kBTile, vb[i]);
      }
      if (kc + 1 < kc_count) load(kc + 1);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (tid == Cfg::kMmaWarp * 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t idesc = instr_desc(NT), a_hi = operand_desc_lo(smem_u32(st)), a_lo = a_hi + (kATileBytes >> 4);
        const uint32_t b_hi = a_hi + (2 * kATileBytes >> 4), b_lo = b_hi + (kBTile >> 4);
#pragma unroll
        for (int ks = 0; ks < kChunkK / 8; ++ks) {
          const uint32_t o = ks * 2, more = kc > 0 || ks > 0;
          mma_tf32_lo(tmem_base + NT, a_lo + o, b_hi + o, idesc, more);
          mma_tf32_lo(tmem_base + NT, a_hi + o, b_lo + o, idesc, 1u);
          mma_tf32_lo(tmem_base, a_hi + o, b_hi + o, idesc, more);
        }
        mma_commit(bars + 8 * stage);
      }
    }
    const bool ok = mbar_wait_abortable(bars + 8 * ((chunk - 1) & 1), (uint32_t)((chunk - 1) >> 1) & 1u, abortp);   // every MMA before it is done too
    if (!__syncthreads_and(ok)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp < 8) {   // two warps per quarter of the lanes, 16 columns in turn
      const int r = (warp & 3) * 32 + lane;
      const bool mine = row0 + r < M && row_marks[r];
      for (int at = (warp >> 2) * 16; at < NT; at += 32) {
        uint32_t v[16], w[16];
        const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)at;
        GTC_TMEM_LD16(v, taddr);
        GTC_TMEM_LD16(w, taddr + (uint32_t)NT);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 16; q += 4)
          if (mine && n0 + at + q < ldc)
            *reinterpret_cast<float4*>(C + (row0 + r) * ldc + n0 + at + q) =
                make_float4(__uint_as_float(v[q]) + __uint_as_float(w[q]), __uint_as_float(v[q + 1]) + __uint_as_float(w[q + 1]),
                            __uint_as_float(v[q + 2]) + __uint_as_float(w[q + 2]), __uint_as_float(v[q + 3]) + __uint_as_float(w[q + 3]));
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();   // the sums and the row marks have been read
  }
  return true;
}

// Roles (see k_gemm_tc_ws; the waits, the abort flag and the way out are the same):
//   copy warp   one thread: raw tile of A by a tensor copy, B's chunk by a bulk copy, into slot j mod R as soon as it is free
//   producers   four or eight warps: scale and split the raw tile of A where it lies (a pair of halves takes the room of its float, and a
//               warp's 16 rows become its own two groups of A_hi and A_lo); arrive on ready[slot]
//   MMA warp    one thread issues; its commit frees the slot
//   epilogue    accumulators -> scales taken off -> C
template <int NT>
__global__ void __launch_bounds__(HalfCfg<NT>::kThreads, 1)
k_gemm_half(const float* __restrict__ A, int lda, const float* __restrict__ row_max, const float* __restrict__ Bk, int ldbk, float* C, int ldc, int M, int N,
            int K, const int* __restrict__ skip, int* __restrict__ error_flag, const uint8_t* __restrict__ b_image, const __grid_constant__ CUtensorMap tmap_a) {
  using Cfg = HalfCfg<NT>;
  constexpr int R = Cfg::kSlots, SETS = Cfg::kSets;
  static_assert(NT <= 256 && NT % 16 == 0, "NT");
  static_assert(Cfg::kSlot % 1024 == 0, "operand tiles start on swizzle boundaries");
  if (skip != nullptr && *skip) return;

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[3 * R + 7];           // raw[R], ready[R], empty[R], acc_full[2], acc_empty[2], drain, redo[2]
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag, copies;                          // copies: chunks whose copies have been started
  __shared__ int redo_some, image_marked;                     // elements too small for a pair in the marked tiles; the image's marks
  __shared__ uint32_t marked[kRedoBits / 32];                 // row tiles with elements too small for a pair
  __shared__ unsigned col_range[2];                           // bits of the largest and, inverted, of the smallest column factor
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar_raw = smem_u32(&bars[0]), bar_ready = smem_u32(&bars[R]), bar_empty = smem_u32(&bars[2 * R]);
  const uint32_t bar_acc_full = smem_u32(&bars[3 * R]), bar_acc_empty = smem_u32(&bars[3 * R + 2]), bar_drain = smem_u32(&bars[3 * R + 4]), bar_redo = smem_u32(&bars[3 * R + 5]);
  constexpr uint32_t kSlot = (uint32_t)Cfg::kSlot, kEpiBase = (uint32_t)R * kSlot;
  float* const col_factor = reinterpret_cast<float*>(smem + kEpiBase + Cfg::kEpiWarps * 4096);   // inverse scales of this CTA's columns

  const int kc_count = (K + kChunkK - 1) / kChunkK;
  if (tid == 0) {
    for (int r = 0; r < R; ++r) { mbar_init(bar_raw + 8 * r, 1); mbar_init(bar_ready + 8 * r, Cfg::kProdWarps); mbar_init(bar_empty + 8 * r, 1); }   // ready: one arrival per producer warp
    for (int a = 0; a < 2; ++a) { mbar_init(bar_acc_full + 8 * a, 1); mbar_init(bar_acc_empty + 8 * a, Cfg::kEpiWarps); }
    mbar_init(bar_drain, 1);
    for (int i = 0; i < 2; ++i) mbar_init(bar_redo + 8 * i, 1);
    abort_flag = copies = redo_some = image_marked = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 2) col_range[tid] = 0u;
  if (tid < kRedoBits / 32) marked[tid] = 0u;
  if (warp == Cfg::kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(Cfg::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = tmem_base_slot;
  volatile int* abortp = &abort_flag;
  const float* const factors = reinterpret_cast<const float*>(b_image + image_blocks_bytes(gridDim.y, NT, kc_count));
  if (warp >= Cfg::kProdWarps && warp < Cfg::kMmaWarp) {   // the epilogue's own; it waits at a barrier of its own below
    for (int c = tid - Cfg::kProdWarps * 32; c < NT; c += Cfg::kEpiWarps * 32) {
      const float f = factors[blockIdx.y * NT + c];
      col_factor[c] = f;
      atomicMax(&col_range[0], __float_as_uint(f));
      atomicMax(&col_range[1], ~__float_as_uint(f));
    }
  }

  const int n_tiles = (M + kBlockM - 1) / kBlockM;
  const int my_tiles = (n_tiles > (int)blockIdx.x) ? (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const int total = my_tiles * kc_count;
  const int n0 = blockIdx.y * NT;

  if (warp < Cfg::kProdWarps) {
    // ---------------- producers ----------------
    // Lane: rows row, row + 8, .. of the tile, eight columns of each (16-byte units 2u, 2u + 1 of the raw row).  Eight raw rows of
    // 128 bytes become 512 bytes of A_hi and 512 of A_lo in their place: nothing outside the warp's own rows is read or written.
    constexpr int GROUPS = kBlockM / 8 / Cfg::kProdWarps;   // of eight rows, per warp
    const int u = lane & 3, row = warp * (8 * GROUPS) + (lane >> 2);
    float ahead[GROUPS];   // row maxima of the next tile
    auto fetch_max = [&](int tile_i) {
#pragma unroll
      for (int i = 0; i < GROUPS; ++i) {
        const long long r = ((long long)blockIdx.x + (long long)tile_i * gridDim.x) * kBlockM + row + 8 * i;
        ahead[i] = tile_i < my_tiles && r < M ? __ldg(row_max + r) : 0.f;
      }
    };
    fetch_max(0);
    int marks = 0;         // the image's, while the first copies are under way
    for (int i = lane; i < image_marks(gridDim.y, NT, kc_count); i += 32) marks |= __ldg(reinterpret_cast<const int*>(factors) + gridDim.y * NT + i);
    marks = (int)__reduce_or_sync(0xffffffffu, (unsigned)marks);
    if (tid == 0) image_marked = marks;
    const bool look = (marks & kWide) != 0;   // always looking takes 256 x 256 on 169 k rows from 88.5 to 92.0 us, 256 x 47 on 2.45 M from 640 to 686
    float scale[GROUPS];
    bool small = false;    // an element of this tile is too small for a pair
    int slot = 0, kc = 0, tile_i = 0;
    uint32_t raw_parity = 0;
    for (int j = 0; j < total; ++j) {
      if (kc == 0) {
#pragma unroll
        for (int i = 0; i < GROUPS; ++i) scale[i] = scale_of(ahead[i]);
        fetch_max(++tile_i);
      }
      if (!__all_sync(0xffffffffu, mbar_wait_abortable(bar_raw + 8 * slot, raw_parity, abortp))) break;   // warp-uniform: the arrival below is per warp
      uint8_t* const tile = smem + (size_t)slot * kSlot;
      float4 a[GROUPS], b[GROUPS];
#pragma unroll
      for (int i = 0; i < GROUPS; ++i) {
        a[i] = *reinterpret_cast<const float4*>(tile + swz(row + 8 * i, 2 * u));
        b[i] = *reinterpret_cast<const float4*>(tile + swz(row + 8 * i, 2 * u + 1));
      }
      __syncwarp();   // all of the warp's rows are in registers
#pragma unroll
      for (int i = 0; i < GROUPS; ++i) {
        uint4 hi, lo;
        split_unit(a[i], b[i], scale[i], hi, lo);
        if (look) small |= least_key(a[i], b[i]) < below_pairs(scale[i]);
        uint8_t* const at = tile + (size_t)(warp * GROUPS + i) * (2 * kHalfGroup) + swz_half(lane >> 2, u);
        *reinterpret_cast<uint4*>(at) = hi;
        *reinterpret_cast<uint4*>(at + kHalfGroup) = lo;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive_warp(bar_ready + 8 * slot);
      if (++kc == kc_count) {
        kc = 0;
        if (small) {
          const int bit = min(tile_i - 1, kRedoBits - 1);
          atomicOr(&marked[bit >> 5], 1u << (bit & 31));
          redo_some = 1;
          small = false;
        }
      }
      if (++slot == R) { slot = 0; raw_parity ^= 1u; }
    }
  } else if (warp == Cfg::kMmaWarp + 1) {
    // ---------------- copies ----------------
    if (lane == 0) {
      constexpr uint32_t b_bytes = (uint32_t)Cfg::kBBytes;
      const uint8_t* const b_src = b_image + (size_t)blockIdx.y * kc_count * b_bytes;
      int kc = 0, tile = blockIdx.x, slot = 0;
      uint32_t empty_parity = 1;   // a fresh barrier passes a wait on parity 1
      for (int j = 0; j < total; ++j) {
        if (!mbar_wait_abortable(bar_empty + 8 * slot, empty_parity, abortp)) break;
        const uint32_t dst_a = smem_base + (uint32_t)slot * kSlot;
        const uint32_t raw_bar = bar_raw + 8 * slot;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(raw_bar), "r"((uint32_t)kATileBytes + b_bytes) : "memory");
        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                     ::"r"(dst_a), "l"(&tmap_a), "r"(kc * kChunkK), "r"(tile * kBlockM), "r"(raw_bar)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(dst_a + (uint32_t)kATileBytes), "l"(b_src + (size_t)kc * b_bytes), "r"(b_bytes), "r"(raw_bar)
                     : "memory");
        copies = j + 1;
        if (++kc == kc_count) { kc = 0; tile += gridDim.x; }
        if (++slot == R) { slot = 0; empty_parity ^= 1u; }
      }
    }
  } else if (warp == Cfg::kMmaWarp) {
    // ---------------- MMA issue: counters that wrap, one addition per operand (see k_gemm_tc_ws) ----------------
    if (lane == 0) {
      const uint32_t idesc = instr_desc_half(NT), idesc2 = instr_desc_half(NT <= 128 ? 2 * NT : NT);
      int kc = 0, tile_i = 0, slot = 0;
      uint32_t ready_parity = 0;
      for (int j = 0; j < total; ++j) {
        const int set = SETS == 1 ? 0 : (tile_i & 1);
        if (kc == 0 && tile_i >= SETS && !mbar_wait_abortable(bar_acc_empty + 8 * set, ((tile_i / SETS) - 1) & 1, abortp)) break;
        // the producers have waited for the slot's copies, B's among them
        if (!mbar_wait_abortable(bar_ready + 8 * slot, ready_parity, abortp)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a_hi = operand_desc_lo(smem_base + slot * kSlot), a_lo = a_hi + (kHalfGroup >> 4);
        const uint32_t b_hi = a_hi + (kATileBytes >> 4), b_lo = b_hi + (NT * kHalfRow >> 4);
        const uint32_t acc = tmem_base + (uint32_t)(set * 2 * NT);
#pragma unroll
        for (int ks = 0; ks < kChunkK / 16; ++ks) {
          const uint32_t o = ks * 2;   // 32 bytes per K step, in 16-byte units
          const uint32_t first = (ks > 0) ? 1u : (kc > 0 ? 1u : 0u);
          if constexpr (NT <= 128) {   // A_hi [B_hi; B_lo]: main product and the first correction in one MMA
            mma_half(acc, a_hi + o, b_hi + o, idesc2, first);
            mma_half(acc + NT, a_lo + o, b_hi + o, idesc, 1u);
          } else {
            mma_half(acc + NT, a_lo + o, b_hi + o, idesc, first);
            mma_half(acc + NT, a_hi + o, b_lo + o, idesc, 1u);
            mma_half(acc, a_hi + o, b_hi + o, idesc, first);
          }
        }
        mma_commit(bar_empty + 8 * slot);
        if (++kc == kc_count) {
          mma_commit(bar_acc_full + 8 * set);
          kc = 0;
          ++tile_i;
        }
        if (++slot == R) { slot = 0; ready_parity ^= 1u; }
      }
    }
  } else {
    // ---------------- epilogue: through a per-warp buffer to whole lines (see k_gemm_tc_ws) ----------------
    const int quarter = warp & 3;
    constexpr int CW = (NT % 32 == 0) ? 32 : 16;
    constexpr int SLOTS = CW / 4;
    constexpr int ROWS_PER_STORE = 32 / SLOTS;
    constexpr int WARPS_PER_QUARTER = Cfg::kEpiWarps / 4, STEPS = NT / CW / WARPS_PER_QUARTER;
    static_assert(NT == STEPS * CW * WARPS_PER_QUARTER, "every column has its step");
    asm volatile("bar.sync 1, %0;" ::"n"(Cfg::kEpiWarps * 32) : "memory");   // the column factors are there
    const float col_most = __uint_as_float(col_range[0]), col_least = __uint_as_float(~col_range[1]);
    const int turn = (warp - Cfg::kProdWarps) >> 2;   // which of the quarter's warps this is: they take the column steps in turn
    uint8_t* tbuf = smem + kEpiBase + (size_t)(warp - Cfg::kProdWarps) * 4096;
    for (int tile_i = 0; tile_i < my_tiles; ++tile_i) {
      const int set = tile_i % SETS;
      const long long row0 = ((long long)blockIdx.x + (long long)tile_i * gridDim.x) * kBlockM + quarter * 32;
      const float row_factor = inverse_scale_of(row0 + lane < M ? __ldg(row_max + row0 + lane) : 0.f);
      if (!__all_sync(0xffffffffu, mbar_wait_abortable(bar_acc_full + 8 * set, (tile_i / SETS) & 1, abortp))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // whether row and column factors may be joined: normal numbers for every pair of the warp's
      const bool joined = __all_sync(0xffffffffu, row_factor * col_most <= 0x1p126f && row_factor * col_least >= 0x1p-126f);
      uint32_t v[16], w[16];   // main product and corrections of 16 columns; with one accumulator set read ahead, beside the stores of those before
      constexpr bool AHEAD = SETS == 1;
      const auto fetch = [&](int part) {   // part of this warp's columns: CW / 16 of them make a step
        const int at = (turn + part / (CW / 16) * WARPS_PER_QUARTER) * CW + part % (CW / 16) * 16;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(set * 2 * NT + at);
        GTC_TMEM_LD16(v, taddr);
        GTC_TMEM_LD16(w, taddr + (uint32_t)NT);
      };
      if (AHEAD) fetch(0);
#pragma unroll 1
      for (int step = 0; step < STEPS; ++step) {
        const int at = (turn + step * WARPS_PER_QUARTER) * CW;   // first column of the step, of this CTA's
#pragma unroll
        for (int half = 0; half < CW / 16; ++half) {
          if (!AHEAD) fetch(step * (CW / 16) + half);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          float sum[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) sum[k] = fmaf(__uint_as_float(w[k]), 1.f / kLoScale, __uint_as_float(v[k]));
          if (half + 1 < CW / 16 || step + 1 < STEPS) {
            if (AHEAD) fetch(step * (CW / 16) + half + 1);
          } else {   // the set is empty
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive_warp(bar_acc_empty + 8 * set);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 f = *reinterpret_cast<const float4*>(col_factor + at + half * 16 + q * 4);
            float4 x = make_float4(sum[q * 4], sum[q * 4 + 1], sum[q * 4 + 2], sum[q * 4 + 3]);
            if (joined) {
              x.x *= row_factor * f.x; x.y *= row_factor * f.y; x.z *= row_factor * f.z; x.w *= row_factor * f.w;
            } else {   // the smaller factor first: the sum times the larger one may leave the range too
              const auto scaled = [&](float y, float c) { return y * fminf(row_factor, c) * fmaxf(row_factor, c); };
              x = make_float4(scaled(x.x, f.x), scaled(x.y, f.y), scaled(x.z, f.z), scaled(x.w, f.w));
            }
            *reinterpret_cast<float4*>(tbuf + lane * 128 + (((half * 4 + q) ^ (lane & (SLOTS - 1))) * 16)) = x;
          }
        }
        __syncwarp();
        const int c4 = lane & (SLOTS - 1);
        const int col = n0 + at + c4 * 4;
#pragma unroll
        for (int i = 0; i < SLOTS; ++i) {
          const int r = i * ROWS_PER_STORE + lane / SLOTS;
          const float4 val = *reinterpret_cast<const float4*>(tbuf + r * 128 + ((c4 ^ (r & (SLOTS - 1))) * 16));
          if (row0 + r < M && col < ldc) *reinterpret_cast<float4*>(C + (row0 + r) * ldc + col) = val;
        }
        __syncwarp();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  const bool gave_up = __syncthreads_or(*abortp);
  const bool all = (image_marked & kBelowPairs) != 0;
  if (!gave_up && (all || redo_some)) {
    redo_rows<NT>(A, lda, row_max, Bk, ldbk, C, ldc, M, N, K, marked, all, smem, tmem_base, bar_redo, abortp);
    __syncthreads();
  }
  if (abort_flag) {
    if (tid == 0) {
      atomicOr(error_flag, 1);
      drain_copies(bar_raw, R, copies);
    }
    if (tid == Cfg::kMmaWarp * 32) drain_mmas(bar_drain);
    __syncthreads();
  }
  if (warp == Cfg::kMmaWarp) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(Cfg::kTmemCols) : "memory");
  }
}

}  // namespace gtc
