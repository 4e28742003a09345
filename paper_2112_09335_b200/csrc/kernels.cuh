// Device kernels of the community-based ADMM GCN trainer (sm_100a).
//
// Layout: every N x C matrix is row-major fp32 with a leading dimension padded to a multiple
// of 4 floats, rows in community order, so that a row starts on a 16-byte boundary and can be
// moved with 128-bit loads.  Padding columns are kept at zero.
// Scalars that decide a step size (descent sums, squared norms) are accumulated in fp64.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_half.cuh"
#include "gemm_tc.cuh"

namespace gk {

constexpr int kCand = 4;        // step-size candidates scored per pass
constexpr int kMaxClassesPerLane = 4;   // C_L <= 128

// Control block of one quadratic-approximation search (one per W_l, one per Z_{l,m}).
struct SearchCtl {
  double t_prev;   // accepted parameter of the previous search (tau_l or theta_{l,m})
  double t_base;   // first candidate of the current pass
  double gg;       // ||grad||^2
  double xx;       // ||x||^2 of the block
  double q;        // (f(x) - f(x+)) / (gg / 2t) at the accepted trial
  float inv_step;  // 1/t of the accepted trial, 0 when the block stays
  int done;        // search finished (accepted, skipped or exhausted)
  int trial;       // accepted trial index, -1 skipped, -2 exhausted
  int pass;        // passes already scored
  float inv_cand[kCand];  // 1/t of the candidates of the current pass
  // W blocks, for the scale of the weights' split images: largest magnitude of the gradient and of W (k_finish_grad)
  float g_max, w_max;
};

// Numbers and flags the host reads back together.
struct Report {
  double obj[8];
  int status;    // bit 0: a NaN or an infinity reached a step-size decision
  int error;     // a bounded wait ran out: 1 in a tensor-core product, kErrGridBarrier in a search
};

__device__ __forceinline__ float relu(float x) { return x > 0.f ? x : 0.f; }

// relu(h) - relu(h - s) without forming h - s when both sides are active, so that a step s far
// below the rounding unit of h still registers exactly.  With pos = max(h, 0) and neg = max(-h, 0)
// (one of them is zero) the drop is min(s + neg, pos): for h > 0 that is min(s, h), for h <= 0 it
// is min(s - h, 0).  The caller forms pos and neg once per element and passes s = k * inv as the
// two factors, so a candidate costs one fused multiply-add and one minimum.
__device__ __forceinline__ float relu_drop(float k, float inv, float neg, float pos) {
  return fminf(fmaf(k, inv, neg), pos);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sums of N values over the block (up to 8 warps), valid in thread 0: all of them in one round, since a round costs two
// barriers and the shuffle latencies whether it carries one value or four.  `sh` holds N * 8 doubles.
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int j = 0; j < N; ++j) sh[j * 8 + w] = v[j];
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = lane < nw ? sh[j * 8 + lane] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  }
}

// Sums over the `count` blocks that left N values each in partial[b * N + ..], by one block: warp j adds value j, lanes strided,
// then the shuffle tree.  total[0 .. N-1] (shared memory) is valid after the barrier at the end.
template <int N>
__device__ __forceinline__ void add_block_sums(const double* partial, int count, double* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int j = w; j < N; j += nw) {
    double t = 0.0;
#pragma unroll 4
    for (int b = lane; b < count; b += 32) t += __ldcg(partial + (size_t)b * N + j);
    t = warp_sum(t);
    if (lane == 0) total[j] = t;
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------------------
// Propagation  out = A~ x,  A~_ij = dinv_i dinv_j on the pattern of A + I (Problem 1).
// Two kernels: k_spmm_wide (a warp per row, more than 64 columns) and k_spmm_sets (narrower operands).
// A warp walks its stored entries one after the other, so a row of thousands of entries (row lengths follow a
// power law) would keep it busy long after the rest of the grid is done.  Rows longer than `long_len` are
// therefore not handled as rows: they come as `n_items` items {row, first entry, one past the last} (first in
// the grid), whose sums go to `scratch` (one row per item).  The row's items are then added up in
// item order: by the last of them to finish (one counter per long row, left at zero), or by k_spmm_long_rows.
// MAPPED: x and out are dense matrices in the caller's row order; node c's row is perm[c], so that no copy of the operand in
// community order and none back is made.  user_col (may be NULL): perm[col[e]] for every entry, for k_spmm_sets one dependent load
// less on the way to the rows of x (24 k rows of 36 entries, 6 columns: 14.9 -> 13.4 us; in k_spmm_wide it disturbed the order of
// the loads: 135 -> 143 us at 128 columns on 169 k rows).
// RELU: out = A~ max(x, 0), so that a forward pass needs no sweep for its activations.
// row_max (may be NULL): the largest magnitude of every row of `out`, which a product of `out` by split halves scales the row by.
// Values are moved in vectors of VEC floats: four wherever rows start on 16-byte boundaries (always inside the
// library), fewer for a caller's matrix of odd width.
// ------------------------------------------------------------------------------------------
template <int VEC> struct Vec;
template <> struct Vec<1> { using T = float; };
template <> struct Vec<2> { using T = float2; };
template <> struct Vec<4> { using T = float4; };

__device__ __forceinline__ float vfma(float w, float x, float a) { return fmaf(w, x, a); }
__device__ __forceinline__ float2 vfma(float w, float2 x, float2 a) { return make_float2(fmaf(w, x.x, a.x), fmaf(w, x.y, a.y)); }
__device__ __forceinline__ float4 vfma(float w, float4 x, float4 a) {
  return make_float4(fmaf(w, x.x, a.x), fmaf(w, x.y, a.y), fmaf(w, x.z, a.z), fmaf(w, x.w, a.w));
}
__device__ __forceinline__ float vscale(float w, float x) { return w * x; }
__device__ __forceinline__ float2 vscale(float w, float2 x) { return make_float2(w * x.x, w * x.y); }
__device__ __forceinline__ float4 vscale(float w, float4 x) { return make_float4(w * x.x, w * x.y, w * x.z, w * x.w); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float4 vadd(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float vxor(unsigned m, float a, int o) { return __shfl_xor_sync(m, a, o); }
__device__ __forceinline__ float2 vxor(unsigned m, float2 a, int o) { return make_float2(vxor(m, a.x, o), vxor(m, a.y, o)); }
__device__ __forceinline__ float4 vxor(unsigned m, float4 a, int o) {
  return make_float4(vxor(m, a.x, o), vxor(m, a.y, o), vxor(m, a.z, o), vxor(m, a.w, o));
}
__device__ __forceinline__ float vrelu(float a) { return relu(a); }
__device__ __forceinline__ float2 vrelu(float2 a) { return make_float2(relu(a.x), relu(a.y)); }
__device__ __forceinline__ float4 vrelu(float4 a) { return make_float4(relu(a.x), relu(a.y), relu(a.z), relu(a.w)); }
__device__ __forceinline__ float vabsmax(float a) { return fabsf(a); }
__device__ __forceinline__ float vabsmax(float2 a) { return fmaxf(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float vabsmax(float4 a) { return fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))); }
__device__ __forceinline__ void vzero(float& a) { a = 0.f; }
__device__ __forceinline__ void vzero(float2& a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ void vzero(float4& a) { a = make_float4(0.f, 0.f, 0.f, 0.f); }

// How the items of the long rows belong together: rows[r] = {row, first item, number of items}; item_row[k] = the entry
// of `rows` item k belongs to; done: one zeroed counter per entry of `rows`.
struct ItemRows {
  const int4* rows;
  const int* item_row;
  int* done;
};

// Called by the G lanes (mask `gmask`, lane `gl`) that have just written item `unit`'s sums to scratch.
template <typename T, int G>
__device__ __forceinline__ void finish_item(const ItemRows& ir, int unit, T* __restrict__ row_out, const T* scratch, int ldv,
                                            unsigned gmask, int gl, float* row_max) {
  const int lr = ir.item_row[unit];
  const int4 whole = ir.rows[lr];
  __threadfence();
  __syncwarp(gmask);
  int done = 0;
  if (gl == 0) done = atomicAdd(ir.done + lr, 1);
  done = __shfl_sync(gmask, done, 0, G);
  if (done + 1 < whole.z) return;
  __threadfence();
  float m = 0.f;
  for (int f = gl; f < ldv; f += G) {
    T s;
    vzero(s);
#pragma unroll 4
    for (int k = 0; k < whole.z; ++k) s = vadd(s, __ldcg(scratch + (long long)(whole.y + k) * ldv + f));
    row_out[f] = s;
    m = fmaxf(m, vabsmax(s));
  }
  if (row_max != nullptr) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(gmask, m, o));
    if (gl == 0) row_max[whole.x] = m;
  }
  if (gl == 0) ir.done[lr] = 0;
}

// A warp per row, NV vectors per lane.  SLICED: operands of more than 32 NV vectors, a warp per row and block of columns
// (blockIdx.y and, past the limit of that, .z): more warps, and one slice of the operand at a time is what L2 has to hold
// (1000 columns on 14 k rows 195 -> 142 us).  Lane t of a group of 32
// stored entries holds column and weight of entry t, handed to the warp by shuffles.  UN neighbours in flight per
// lane: the kernel is bound by load latency at what its 40 or so resident warps keep in flight (256 columns, 47 entries a row: half of
// the L2-to-SM fabric's peak, L2 58 %, issue slots 46 %; 128 columns, 15 a row: 28, 35 and 54 %), on operands far larger than L2 by DRAM.
// 11 % of the sectors are L1 hits, and yet loads that do not allocate there take 10.4 instead of 6.8 ms (2.45 M rows at 256 columns).
// How the compiler orders the loads counts for as much (the plain loop is faster than one that fetches columns ahead: 118 against 143 us at 128 columns on 169 k rows).
// The bound of 21 blocks gives the 40 registers of 24 and an order of loads that the row maxima at the end do not disturb: 6.81 ms with
// them, 6.75 without; under a bound of 24 blocks 8.78.  With ReLU on the gathered rows it is a bound of 20 (9.0 against 9.4 ms).
template <int VEC, int NV, int UN, bool MAPPED, bool SLICED, bool RELU>
__global__ void __launch_bounds__(64, VEC == 4 ? (RELU ? 20 : 21) : 16)
k_spmm_wide(const int* __restrict__ row_ptr, const int* __restrict__ col, const float* __restrict__ dinv,
            const int* __restrict__ perm, const int4* __restrict__ items, int n, int n_items, int long_len,
            const typename Vec<VEC>::T* __restrict__ x, typename Vec<VEC>::T* __restrict__ out, int ldv,
            typename Vec<VEC>::T* __restrict__ scratch, float* __restrict__ row_max) {
  using T = typename Vec<VEC>::T;
  const int lane = threadIdx.x & 31;
  const int off = SLICED ? (blockIdx.y + gridDim.y * blockIdx.z) * (32 * NV) : 0;
  const int wv = SLICED ? min(32 * NV, ldv - off) : ldv;   // this block's columns
  if (SLICED) { x += off; out += off; scratch += off; }
  const int unit = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (unit >= n + n_items) return;
  int row, rs, re;
  T* dst;
  const bool item = unit < n_items;
  if (item) {
    const int4 it = items[unit];
    row = it.x; rs = it.y; re = it.z;
    dst = scratch + (long long)unit * ldv;
  } else {
    row = unit - n_items;
    rs = row_ptr[row]; re = row_ptr[row + 1];
    if (re - rs > long_len) return;
    dst = out + (long long)(MAPPED ? perm[row] : row) * ldv;
  }
  const float di = dinv[row];
  // The unit once more, behind the compiler's back: kept from above it is a register too many during the walk.
  const auto again = [] {
    unsigned block, thread;
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(block));
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(thread));
    return (int)((block * 64ull + thread) >> 5);
  };
  // One turn only, but the compiler is not to know: it then issues all loads of a step before the first sum (+20 % at 256 columns).
  for (int cb = 0; cb < wv; cb += 32 * NV) {
    T acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) vzero(acc[v]);
    for (int base = rs; base < re; base += 32) {
      int r = 0;
      float w = 0.f;
      if (base + lane < re) {
        const int c = col[base + lane];
        w = dinv[c];
        r = MAPPED ? perm[c] : c;
      }
      const int cnt = min(32, re - base);
      for (int t = 0; t < cnt; t += UN) {
        int rj[UN];
        float wj[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {   // lanes past the row's end hold (row 0, weight 0)
          rj[u] = __shfl_sync(0xffffffffu, r, (t + u) & 31);
          wj[u] = __shfl_sync(0xffffffffu, w, (t + u) & 31);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int f = cb + lane + 32 * v;
          if (f < wv) {
            T xv[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) xv[u] = __ldg(x + (long long)rj[u] * ldv + f);
#pragma unroll
            for (int u = 0; u < UN; ++u) acc[v] = vfma(wj[u], RELU ? vrelu(xv[u]) : xv[u], acc[v]);
          }
        }
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int f = cb + lane + 32 * v;
      if (f < wv) dst[f] = vscale(di, acc[v]);
    }
    if (!MAPPED && !SLICED && row_max != nullptr) {
      float m = 0.f;
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (cb + lane + 32 * v < wv) m = fmaxf(m, vabsmax(acc[v]));
      m = di * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
      const int own = again() - n_items;
      if (lane == 0 && own >= 0) row_max[own] = m;
    }
  }
}

// Rows that k_spmm_wide handled as items (a kernel of its own: with finish_item at its end k_spmm_wide takes more
// registers and was 4 % slower): out[row] = sum of the row's item sums, in item order, one block per row.
template <typename T, bool MAPPED>
__global__ void __launch_bounds__(64)
k_spmm_long_rows(const int4* __restrict__ rows, const T* __restrict__ scratch, T* __restrict__ out, int ldv,
                                 const int* __restrict__ perm, float* __restrict__ row_max) {
  gtc::enter_kernel();
  const int4 r = rows[blockIdx.x];
  const long long row = MAPPED ? perm[r.x] : r.x;
  float m = 0.f;
  for (int f = threadIdx.x; f < ldv; f += blockDim.x) {
    T s;
    vzero(s);
#pragma unroll 4
    for (int k = 0; k < r.z; ++k) s = vadd(s, scratch[(long long)(r.y + k) * ldv + f]);
    out[row * ldv + f] = s;
    m = fmaxf(m, vabsmax(s));
  }
  if (MAPPED || row_max == nullptr) return;
  __shared__ float s_max;
  m = warp_max(m);
  if (threadIdx.x == 32) s_max = m;
  __syncthreads();
  if (threadIdx.x == 0) row_max[row] = fmaxf(m, s_max);
}

// Narrow operands.  G = CL * EP lanes share a row: CL of them side by side over its columns (NV vectors each), EP
// such sets over its stored entries (entry e goes to set (e - first) mod EP), so that a row of k entries costs
// k / EP dependent steps instead of k and a narrow row still fills the lanes of a warp; a shuffle tree adds the
// sets at the end.  The order of a row's sum depends on EP alone: all layouts of a width agree bit for bit.
// CL <= 4: every lane loads column and weight of its own entries (one word for the CL lanes of a set), one step
// ahead of the operand rows.  CL >= 8: the G lanes load one entry each, columns two groups ahead and weights one,
// and hand them to the sets by shuffles (with more lanes per set the repeated loads cost more than the shuffles).
// Rows sharing a warp are taken by falling length, from row_table[k] = {row, first entry, one past the last, dinv}: one load where
// order, row pointers and weight would be two that wait for each other.  Measured at 4 / 16 / 48 columns against one set per row:
// 2.4 M rows, 126 M entries: 5.5 -> 1.1 ms, 2.2 -> 1.0, 2.7 -> 2.7; 13.8 k rows, 0.43 M entries: 293 -> 15 us, 85 -> 15, 37 -> 25.
template <int VEC, int NV, int CL, int EP, int UN, bool MAPPED, bool RELU>
__global__ void __launch_bounds__(128, CL >= 8 && VEC == 4 ? 10 : 8)
k_spmm_sets(const int* __restrict__ row_ptr, const int* __restrict__ col, const float* __restrict__ dinv,
            const int* __restrict__ perm, const int* __restrict__ user_col, const int4* __restrict__ items, int n, int n_items, int long_len,
            const typename Vec<VEC>::T* __restrict__ x, typename Vec<VEC>::T* __restrict__ out, int ldv,
            typename Vec<VEC>::T* __restrict__ scratch, const int4* __restrict__ row_table, const ItemRows ir, float* __restrict__ row_max) {
  gtc::enter_kernel();
  using T = typename Vec<VEC>::T;
  constexpr int G = CL * EP;
  static_assert(G <= 32, "a row is handled inside one warp");
  static_assert(CL <= 4 || UN <= CL, "a group of G entries is CL steps of EP");
  const int lane = threadIdx.x & 31, gl = lane & (G - 1), cl = gl & (CL - 1), set = gl / CL;
  const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << (G & 31)) - 1u) << (lane & ~(G - 1)));
  const int unit = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) / G);
  if (unit >= n + n_items) return;
  int row, rs, re;
  float di;
  const bool item = unit < n_items;
  if (item) {
    const int4 it = items[unit];
    row = it.x; rs = it.y; re = it.z;
    di = dinv[row];
  } else if (G < 32) {
    const int4 it = row_table[unit - n_items];
    row = it.x; rs = it.y; re = it.z;
    di = __int_as_float(it.w);
  } else {
    row = unit - n_items;
    rs = row_ptr[row]; re = row_ptr[row + 1];
    di = dinv[row];
  }
  if (!item && re - rs > long_len) return;
  T* const row_out = out + (long long)(MAPPED ? perm[row] : row) * ldv;
  T* const dst = item ? scratch + (long long)unit * ldv : row_out;
  float m = 0.f;
  for (int cb = 0; cb < ldv; cb += CL * NV) {
    T acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) vzero(acc[v]);
    if constexpr (CL <= 4) {
      int c[UN], ru[UN];
      const auto fetch = [&](int e) {
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          c[u] = (e + u * EP < re) ? col[e + u * EP] : -1;
          if (MAPPED && user_col != nullptr) ru[u] = (e + u * EP < re) ? user_col[e + u * EP] : -1;
        }
      };
      fetch(rs + set);
      for (int e = rs + set; e < re; e += EP * UN) {
        float w[UN];
        int r[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          w[u] = c[u] >= 0 ? dinv[c[u]] : 0.f;
          r[u] = c[u] < 0 || !MAPPED ? c[u] : user_col != nullptr ? ru[u] : perm[c[u]];
        }
        fetch(e + EP * UN);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int f = cb + cl + CL * v;
          if (f < ldv) {
            T xv[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u)
              if (r[u] >= 0) xv[u] = __ldg(x + (long long)r[u] * ldv + f);
#pragma unroll
            for (int u = 0; u < UN; ++u)
              if (r[u] >= 0) acc[v] = vfma(w[u], RELU ? vrelu(xv[u]) : xv[u], acc[v]);
          }
        }
      }
    } else {
      int c_n = rs + gl < re ? col[rs + gl] : -1, c_n2 = rs + G + gl < re ? col[rs + G + gl] : -1;
      const auto row_of = [&](int c, int e) { return c < 0 ? 0 : !MAPPED ? c : user_col != nullptr ? user_col[e] : perm[c]; };
      float w_n = c_n >= 0 ? dinv[c_n] : 0.f;
      int r_n = row_of(c_n, rs + gl);
      for (int base = rs; base < re; base += G) {
        const float w = w_n;
        const int r = r_n;
        c_n = c_n2;
        c_n2 = base + 2 * G + gl < re ? col[base + 2 * G + gl] : -1;
        w_n = c_n >= 0 ? dinv[c_n] : 0.f;
        r_n = row_of(c_n, base + G + gl);
        const int steps = (min(G, re - base) + EP - 1) / EP;
        for (int t = 0; t < steps; t += UN) {
          int rj[UN];
          float wj[UN];
#pragma unroll
          for (int u = 0; u < UN; ++u) {   // lanes past the row's end hold (row 0, weight 0)
            const int src = ((t + u) * EP + set) & (G - 1);
            rj[u] = __shfl_sync(gmask, r, src, G);
            wj[u] = __shfl_sync(gmask, w, src, G);
          }
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const int f = cb + cl + CL * v;
            if (f < ldv) {
              T xv[UN];
#pragma unroll
              for (int u = 0; u < UN; ++u) xv[u] = __ldg(x + (long long)rj[u] * ldv + f);
#pragma unroll
              for (int u = 0; u < UN; ++u) acc[v] = vfma(wj[u], RELU ? vrelu(xv[u]) : xv[u], acc[v]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int o = CL; o < G; o <<= 1)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = vadd(acc[v], vxor(gmask, acc[v], o));
    if (set == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int f = cb + cl + CL * v;
        if (f < ldv) {
          const T s = vscale(di, acc[v]);
          dst[f] = s;
          m = fmaxf(m, vabsmax(s));
        }
      }
    }
  }
  if (item) {
    finish_item<T, G>(ir, unit, row_out, scratch, ldv, gmask, gl, MAPPED ? nullptr : row_max);
  } else if (!MAPPED && row_max != nullptr) {
#pragma unroll
    for (int o = CL / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(gmask, m, o));
    if (gl == 0) row_max[row] = m;
  }
}

// ------------------------------------------------------------------------------------------
// Dense products.
//   k_gemm_nn : C[M x N] = A[M x K] B[K x N]          (H = P W, D = P grad, G = S W^T, T = G W)
//   k_gemm_tn : part[s][Ka x Nb] = sum over the rows of split s of A[r,:]^T B[r,:]   (grad = P^T R)
// fp32 FFMA register tiles; `skip`, when given, points at a flag that cancels the launch.
// ------------------------------------------------------------------------------------------
template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), 2)
k_gemm_nn(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
          float* __restrict__ C, int ldc, int M, int N, int K, const int* __restrict__ skip) {
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int TX = BN / TN;
  constexpr int A_F4 = BM * BK / 4, B_F4 = BK * BN / 4;
  constexpr int A_PER = (A_F4 + NT - 1) / NT, B_PER = (B_F4 + NT - 1) / NT;
  constexpr int PAD = 4;
  static_assert(TN == 4 || TN == 8, "TN");
  static_assert(TM == 4 || TM == 8, "TM");
  if (skip != nullptr && *skip) return;
  __shared__ __align__(16) float As[2][BK][BM + PAD];
  __shared__ __align__(16) float Bs[2][BK][BN];
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const long long row0 = (long long)blockIdx.x * BM;
  const int col0 = blockIdx.y * BN;

  float4 ra[A_PER], rb[B_PER];
  auto load_tiles = [&](int k0) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      const int f = tid + i * NT;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (f < A_F4) {
        const int r = f / (BK / 4), kq = (f % (BK / 4)) * 4;
        const long long gr = row0 + r;
        const int gk = k0 + kq;
        if (gr < M && gk < K) {
          v = *reinterpret_cast<const float4*>(A + gr * lda + gk);   // lda % 4 == 0, gk % 4 == 0
          if (gk + 1 >= K) v.y = 0.f;
          if (gk + 2 >= K) v.z = 0.f;
          if (gk + 3 >= K) v.w = 0.f;
        }
      }
      ra[i] = v;
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      const int f = tid + i * NT;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (f < B_F4) {
        const int kr = f / (BN / 4), c = (f % (BN / 4)) * 4;
        const int gk = k0 + kr, gc = col0 + c;
        if (gk < K && gc < N) {
          v = *reinterpret_cast<const float4*>(B + (long long)gk * ldb + gc);  // ldb % 4 == 0
          if (gc + 1 >= N) v.y = 0.f;
          if (gc + 2 >= N) v.z = 0.f;
          if (gc + 3 >= N) v.w = 0.f;
        }
      }
      rb[i] = v;
    }
  };
  auto store_tiles = [&](int buf) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      const int f = tid + i * NT;
      if (f < A_F4) {
        const int r = f / (BK / 4), kq = (f % (BK / 4)) * 4;
        As[buf][kq + 0][r] = ra[i].x;
        As[buf][kq + 1][r] = ra[i].y;
        As[buf][kq + 2][r] = ra[i].z;
        As[buf][kq + 3][r] = ra[i].w;
      }
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      const int f = tid + i * NT;
      if (f < B_F4) {
        const int kr = f / (BN / 4), c = (f % (BN / 4)) * 4;
        *reinterpret_cast<float4*>(&Bs[buf][kr][c]) = rb[i];
      }
    }
  };

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  load_tiles(0);
  store_tiles(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    const bool more = (k0 + BK) < K;
    if (more) load_tiles(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&As[buf][k][ty * TM + i]);
        a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
      }
      {
        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
        b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
      }
      if constexpr (TN == 8) {
        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][k][BN / 2 + tx * 4]);
        b[TN - 4] = v.x; b[TN - 3] = v.y; b[TN - 2] = v.z; b[TN - 1] = v.w;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      store_tiles(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
  // columns N..ldc-1 (padding) receive the zeros accumulated from the masked B columns
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const long long gr = row0 + ty * TM + i;
    if (gr >= M) continue;
#pragma unroll
    for (int h = 0; h < TN / 4; ++h) {
      const int gc = col0 + (h == 0 ? tx * 4 : BN / 2 + tx * 4);
      if (gc < ldc)
        *reinterpret_cast<float4*>(C + gr * ldc + gc) =
            make_float4(acc[i][h * 4], acc[i][h * 4 + 1], acc[i][h * 4 + 2], acc[i][h * 4 + 3]);
    }
  }
}

// Residuals with respect to the pre-activation H (derivatives of phi, Section 3):
//   hidden layer  R = nu (f(H) - Z) * f'(H)
//   last layer    R = -(U + rho (Z - H))
__device__ __forceinline__ float4 resid_hidden(const float4& h, const float4& z, float nu) {
  return make_float4(h.x > 0.f ? nu * (h.x - z.x) : 0.f, h.y > 0.f ? nu * (h.y - z.y) : 0.f,
                     h.z > 0.f ? nu * (h.z - z.z) : 0.f, h.w > 0.f ? nu * (h.w - z.w) : 0.f);
}
__device__ __forceinline__ float4 resid_out(const float4& h, const float4& z, const float4& u, float rho) {
  return make_float4(-(u.x + rho * (z.x - h.x)), -(u.y + rho * (z.y - h.y)), -(u.z + rho * (z.z - h.z)), -(u.w + rho * (z.w - h.w)));
}

// RESID: B is not stored; it is the hidden layer's R, formed from H (passed as B) and Z (Zres) as they are loaded.
// part[(split * Ka + ka) * ldp + nb].  A: rows x Ka (lda), B: rows x Nb (ldb).
// Split s owns rows [s * rows_per_split, min(rows, (s+1) * rows_per_split)).
template <int BM, int BN, int BK, int TM, int TN, bool RESID>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), 2)
k_gemm_tn(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
          float* __restrict__ part, int ldp, long long rows, long long rows_per_split, int Ka, int Nb, const float* __restrict__ Zres, float nu) {
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int TX = BN / TN;
  constexpr int A_F4 = BK * BM / 4, B_F4 = BK * BN / 4;
  constexpr int A_PER = (A_F4 + NT - 1) / NT, B_PER = (B_F4 + NT - 1) / NT;
  static_assert(TM == 4 || TM == 8, "TM");
  static_assert(BN % 4 == 0, "BN");
  __shared__ __align__(16) float As[2][BK][BM];
  __shared__ __align__(16) float Bs[2][BK][BN];
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int a0 = blockIdx.x * BM, b0 = blockIdx.y * BN;
  const long long r_begin = (long long)blockIdx.z * rows_per_split;
  const long long r_end = min(rows, r_begin + rows_per_split);

  float4 ra[A_PER], rb[B_PER];
  auto load_tiles = [&](long long r0) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      const int f = tid + i * NT;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (f < A_F4) {
        const int rr = f / (BM / 4), c = (f % (BM / 4)) * 4;
        const long long gr = r0 + rr;
        const int gc = a0 + c;
        if (gr < r_end && gc < Ka) {
          v = *reinterpret_cast<const float4*>(A + gr * lda + gc);
          if (gc + 1 >= Ka) v.y = 0.f;
          if (gc + 2 >= Ka) v.z = 0.f;
          if (gc + 3 >= Ka) v.w = 0.f;
        }
      }
      ra[i] = v;
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      const int f = tid + i * NT;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (f < B_F4) {
        const int rr = f / (BN / 4), c = (f % (BN / 4)) * 4;
        const long long gr = r0 + rr;
        const int gc = b0 + c;
        if (gr < r_end && gc < Nb) {
          v = *reinterpret_cast<const float4*>(B + gr * ldb + gc);
          if (RESID) v = resid_hidden(v, *reinterpret_cast<const float4*>(Zres + gr * ldb + gc), nu);
          if (gc + 1 >= Nb) v.y = 0.f;
          if (gc + 2 >= Nb) v.z = 0.f;
          if (gc + 3 >= Nb) v.w = 0.f;
        }
      }
      rb[i] = v;
    }
  };
  auto store_tiles = [&](int buf) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      const int f = tid + i * NT;
      if (f < A_F4) *reinterpret_cast<float4*>(&As[buf][f / (BM / 4)][(f % (BM / 4)) * 4]) = ra[i];
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      const int f = tid + i * NT;
      if (f < B_F4) *reinterpret_cast<float4*>(&Bs[buf][f / (BN / 4)][(f % (BN / 4)) * 4]) = rb[i];
    }
  };

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  if (r_begin < r_end) {
    load_tiles(r_begin);
    store_tiles(0);
    __syncthreads();
    int buf = 0;
    for (long long r0 = r_begin; r0 < r_end; r0 += BK) {
      const bool more = (r0 + BK) < r_end;
      if (more) load_tiles(r0 + BK);
#pragma unroll
      for (int k = 0; k < BK; ++k) {
        float a[TM], b[TN];
        {
          const float4 v = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]);
          a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
        }
        if constexpr (TM == 8) {
          const float4 v = *reinterpret_cast<const float4*>(&As[buf][k][BM / 2 + ty * 4]);
          a[TM - 4] = v.x; a[TM - 3] = v.y; a[TM - 2] = v.z; a[TM - 1] = v.w;
        }
        if constexpr (TN >= 4) {
          const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
          b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
          if constexpr (TN == 8) {
            const float4 w = *reinterpret_cast<const float4*>(&Bs[buf][k][BN / 2 + tx * 4]);
            b[TN - 4] = w.x; b[TN - 3] = w.y; b[TN - 2] = w.z; b[TN - 1] = w.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < TN; ++j) b[j] = Bs[buf][k][tx * TN + j];
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
      if (more) {
        store_tiles(buf ^ 1);
        __syncthreads();
        buf ^= 1;
      }
    }
  }
  float* dst = part + (long long)blockIdx.z * Ka * ldp;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int ga = a0 + ((TM == 8 && i >= 4) ? BM / 2 + ty * 4 + (i - 4) : ty * 4 + i);
    if (ga >= Ka) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int gb;
      if (TN == 8) gb = b0 + (j >= 4 ? BN / 2 + tx * 4 + (j - 4) : tx * 4 + j);
      else if (TN == 4) gb = b0 + tx * 4 + j;
      else gb = b0 + tx * TN + j;
      if (gb < ldp) dst[(long long)ga * ldp + gb] = acc[i][j];
    }
  }
}

// ------------------------------------------------------------------------------------------
// Residuals where they are stored.
// ------------------------------------------------------------------------------------------
__global__ void k_resid_hidden(const float4* __restrict__ H, const float4* __restrict__ Z,
                               float4* __restrict__ R, long long n4, float nu) {
  gtc::enter_kernel();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (long long)gridDim.x * blockDim.x)
    R[i] = resid_hidden(H[i], Z[i], nu);
}

__global__ void k_resid_out(const float4* __restrict__ H, const float4* __restrict__ Z,
                            const float4* __restrict__ U, float4* __restrict__ R, long long n4, float rho) {
  gtc::enter_kernel();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (long long)gridDim.x * blockDim.x)
    R[i] = resid_out(H[i], Z[i], U[i], rho);
}

// ------------------------------------------------------------------------------------------
// Step-size searches (Section 3.1 for W, Eq. 9 for Z).  A search is one cooperative launch: score candidates, add the
// blocks' sums up in a fixed order, decide, score again while a search is open, then move the block.  As separate
// launches (ten sweeps of scoring and decision, nine of which usually found nothing to do) this was half of the
// kernels of a pass and, on graphs of a few thousand nodes, most of its time.
// ------------------------------------------------------------------------------------------
// Grid-wide rendezvous of a cooperative launch (all blocks resident).  Every wait is bounded by elapsed clocks (a few
// seconds); one that runs out raises *err and every block leaves the kernel.  A launch that finds *err raised (by itself or by
// any launch before it) leaves at once: the counters between launches, this one among them, may then hold anything until the
// host has seen the flag and zeroed them.
struct GridBar {
  unsigned arrived, generation;
};
constexpr int kErrGridBarrier = 2;
constexpr long long kGridWaitClocks = 1LL << 33;

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits until every block of the grid has arrived; the last one to arrive runs `last` (with all its threads) before
// the others are let go.  What blocks wrote before the call is visible to `last`, and what `last` wrote to everyone after it.
// False when the wait ran out (the same in every thread of the block).
template <typename F>
__device__ __forceinline__ bool grid_meet(GridBar* bar, int* err, F&& last) {
  __shared__ int s_last, s_ok;
  __syncthreads();
  unsigned gen = 0;
  if (threadIdx.x == 0) {
    gen = load_acquire(&bar->generation);
    __threadfence();
    s_last = atomicAdd(&bar->arrived, 1u) == gridDim.x - 1;
    s_ok = 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    last();
    __syncthreads();
    if (threadIdx.x == 0) {
      bar->arrived = 0;
      __threadfence();
      store_release(&bar->generation, gen + 1);
    }
  } else if (threadIdx.x == 0) {
    const long long t0 = clock64();
    for (unsigned i = 1; load_acquire(&bar->generation) == gen; ++i) {
      if ((i & 63u) == 0u && __ldcg(err) != 0) { s_ok = 0; break; }   // others have left or will not come
      if (clock64() - t0 > kGridWaitClocks) { s_ok = 0; atomicOr(err, kErrGridBarrier); break; }
    }
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ __forceinline__ void set_candidates(SearchCtl* c, double growth) {
  double t = c->t_base;
#pragma unroll
  for (int j = 0; j < kCand; ++j) { c->inv_cand[j] = (float)(1.0 / t); t *= growth; }
}

// Starts one search from ||grad||^2 and ||x||^2 of its block.
__device__ __forceinline__ void begin_one(SearchCtl* c, double gg, double xx, double shrink, double growth,
                                          int* __restrict__ n_active, int* __restrict__ status) {
  c->gg = gg;
  c->xx = xx;
  c->pass = 0;
  c->q = 0.0;
  c->inv_step = 0.f;
  if (!(c->gg > 1e-24 * c->xx)) {          // zero up to rounding (also catches NaN): skip
    c->done = 1;
    const bool finite = (c->gg == c->gg) && (c->xx == c->xx) && c->gg < 1.0e300 && c->xx < 1.0e300;
    c->trial = finite ? -1 : -2;
    if (!finite) atomicOr(status, 1);     // a NaN or an infinity reached the gradient or the block itself
    return;
  }
  c->done = 0;
  c->trial = -2;
  c->t_base = fmax(c->t_prev * shrink, 1e-12);
  set_candidates(c, growth);
  if (n_active) atomicAdd(n_active, 1);
}

// One decision per search.  mode 0: `cand` sums of a scoring pass, delta_j = scale * sum[j]
// plus the quadratic own term; mode 1: closed form, delta(t) = -lin/t + quad/t^2, all trials at once.
//   own term (Z blocks only): -(nu/t) sag + (nu/2t^2) sgg with sag = <Z - f(H), G>, sgg = gg
struct DecideArgs {
  double growth;
  int max_trials;
  int mode;          // 0 scored candidates, 1 closed form
  int cand;          // mode 0: candidates scored per pass (<= kCand)
  double scale;      // multiplies the scored sums (nu/2)
  double quad_coef;  // closed form: delta = -sum[0]/t + quad_coef * sum[1] / t^2
  double own_nu;     // nu when the block has a quadratic own term, else 0
};

// Decision of one open search from the sums of the sweep just scored, by the 32 lanes of a warp (sums, sag the same in
// all): lane j tries the j-th trial, t = t_base * growth^j, and the first lane whose trial meets the condition
// f(x+) - f(x) <= -||g||^2 / (2t) has its trial accepted.  The fp64 divisions of a trial are a chain of several hundred
// clocks; one after the other they were most of a small search.  Returns true when the search goes on to another sweep
// (its candidates are then already set).
__device__ __forceinline__ bool decide_one(SearchCtl* c, const double* sums, double sag, const DecideArgs& a, int* n_active,
                                           int* status) {
  const int lane = threadIdx.x & 31;
  const double gg = c->gg, t_base = c->t_base;
  const int first = a.mode == 1 ? 0 : c->pass * a.cand;
  const int tries = min(a.mode == 1 ? a.max_trials : a.cand, a.max_trials - first);
  const double lin = a.mode == 1 ? sums[0] : 0.0, quad = a.mode == 1 ? a.quad_coef * sums[1] : 0.0;
  double t = t_base;
  for (int j = 0; j < (lane < tries ? lane : 0); ++j) t *= a.growth;
  int found = -1;
  double delta = 0.0, need = 1.0;
  bool finite = true;
  for (int base = 0; base < tries && found < 0; base += 32) {
    const int j = base + lane;
    bool pass = false;
    if (j < tries) {
      const double own = 0.5 * a.own_nu * gg / (t * t) - a.own_nu * sag / t;
      if (a.mode == 1) delta = -lin / t + quad / (t * t) + own;
      else {
        const double sum = sums[j & (kCand - 1)];
        finite = sum == sum;
        delta = a.scale * sum + own;
      }
      need = gg / (2.0 * t);
      pass = delta <= -need;         // false for NaN
    }
    const unsigned hits = __ballot_sync(0xffffffffu, pass);
    if (hits != 0u) found = base + __ffs((int)hits) - 1;
    else if (base + 32 < tries)
      for (int k = 0; k < 32; ++k) t *= a.growth;
  }
  if (a.mode == 1) finite = lin == lin && quad == quad;
  // trials behind the accepted one are not looked at: their sums may be anything
  const unsigned bad = __ballot_sync(0xffffffffu, !finite);
  const bool nonfinite = a.mode == 1 ? (bad != 0u && found < 0) : (bad & (found < 0 ? 0xffffffffu : (2u << (found & 31)) - 1u)) != 0u;
  bool goes_on = false;
  if (found >= 0) {
    if (lane == (found & 31)) {
      c->t_prev = t;
      c->q = -delta / need;
      c->inv_step = (float)(1.0 / t);
      c->trial = first + found;
      c->done = 1;
    }
  } else {
    goes_on = a.mode == 0 && first + a.cand < a.max_trials;
    double next = t_base;
    if (goes_on)
      for (int j = 0; j < a.cand; ++j) next *= a.growth;
    if (lane == 0) {
      if (a.mode == 0) c->pass += 1;
      if (goes_on) { c->t_base = next; set_candidates(c, a.growth); }
      else { c->done = 1; c->trial = -2; c->inv_step = 0.f; }
    }
  }
  if (lane == 0) {
    if (nonfinite) atomicOr(status, 1);
    if (!goes_on && n_active) atomicSub(n_active, 1);
  }
  __syncwarp();
  return goes_on;
}

// The decision log is a ring of `ring` passes; the slot in use is *pass mod ring, with the pass counter
// kept on the device so that a recorded launch sequence stays valid from one pass to the next.
struct DecisionLog {
  int* trial;
  double* q;
  const int* pass;
  long long per_pass, offset;   // entries of a pass, first entry of this block family
  int ring;
};
__device__ __forceinline__ void log_decision(const DecisionLog& lg, int i, const SearchCtl* c) {
  const long long at = (long long)(*lg.pass % lg.ring) * lg.per_pass + lg.offset + i;
  lg.trial[at] = c->trial;
  lg.q[at] = c->q;
}

// Weight matrices are written in two orders at once (themselves and their transpose, a split image for either): in tiles of 32 x
// 32 that turn through shared memory, because a column of single floats costs a memory sector per element.
// `value(r, c)` is called once per element of the tile, padding columns included, and gives its new value; t may be NULL.  The
// transpose's padding columns are written too: layers of other sizes share the buffer of the gradient's.
// Blocks of 256 threads, all of them.
using WeightTile = float[32][33];
template <typename F>
__device__ __forceinline__ void weight_tile(int tile, int rows, int cols, int padded, WeightTile& turn, float* __restrict__ t, int ldt,
                                            const gtc::Image& image, const gtc::Image& image_t, float scale, F&& value) {
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, col_tiles = (padded + 31) / 32;
  const int r0 = tile / col_tiles * 32, c0 = tile % col_tiles * 32;
  __syncthreads();   // the tile before this one has been read
#pragma unroll
  for (int k = 0; k < 32; k += 8) {
    const int r = r0 + y + k, c = c0 + x;
    if (r < rows && c < padded) {
      const float v = value(r, c);
      turn[y + k][x] = v;
      if (c < cols) gtc::put_half(image_t, r, c, v * scale);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 32; k += 8) {
    const int r = r0 + x, c = c0 + y + k;
    if (c >= cols) continue;
    if (r < rows) {
      const float v = turn[x][y + k];
      if (t != nullptr) t[(long long)c * ldt + r] = v;
      gtc::put_half(image, c, r, v * scale);
    } else if (t != nullptr && r < ldt) {
      t[(long long)c * ldt + r] = 0.f;
    }
  }
}

// Weight gradient from its split partial sums, and the start of the W_l search, in one launch:
//   grad[e] = sum over splits of part[s][e] (fp64, in split order), its transpose for P grad, ||grad||^2 and ||W||^2.  `maxima`: the
//   largest magnitudes of grad and W go to the control block, for the images of W after its move.
// SG = 1: a block owns a tile of 32 x 32 elements (grid: tiles over rows x ldp).  SG = 8 (many splits): 32 consecutive elements,
// eight threads per element, each adding its own run of consecutive splits; the transpose is then written one
// float at a time (a tile of 32 x 32 would leave one block where there are 32 now).  The last block to finish adds the
// blocks' sums of squares up in block order and starts the search.  W = NULL: only the sum over the splits.
template <int SG>
__global__ void __launch_bounds__(256)
k_finish_grad(const float* __restrict__ part, int splits, int rows, int cols, int ldp, float* __restrict__ grad,
              float* __restrict__ grad_t, int ldt, const float* __restrict__ W, double* partial, unsigned* ticket,
              SearchCtl* ctl, double shrink, double growth, int* status, bool maxima) {
  gtc::enter_kernel();
  __shared__ double sh[16], s_part[SG == 1 ? 1 : SG][32];
  __shared__ WeightTile turn;
  __shared__ int s_last;
  const long long elems = (long long)rows * ldp;
  double sq[2] = {0.0, 0.0};   // of grad, of W
  float most[2] = {0.f, 0.f};
  const auto sum_splits = [&](long long e, int k0, int k1) {
    double s = 0.0;
#pragma unroll 8
    for (int k = k0; k < k1; ++k) s += (double)part[k * elems + e];
    return s;
  };
  if (SG == 1) {
    weight_tile((int)blockIdx.x, rows, cols, ldp, turn, W != nullptr ? grad_t : nullptr, ldt, gtc::Image{nullptr, 16, 1}, gtc::Image{nullptr, 16, 1}, 1.f, [&](int r, int c) {
      const long long e = (long long)r * ldp + c;
      const float g = (float)sum_splits(e, 0, splits);
      grad[e] = g;
      if (W != nullptr) {
        const float w = W[e];
        sq[0] += (double)g * (double)g; sq[1] += (double)w * (double)w;
        most[0] = fmaxf(most[0], fabsf(g)); most[1] = fmaxf(most[1], fabsf(w));
      }
      return g;
    });
  } else {
    const int x = threadIdx.x & 31, sg = threadIdx.x >> 5;
    const long long e = (long long)blockIdx.x * 32 + x;
    const bool in = e < elems;
    const float w = in && W != nullptr && sg == 0 ? W[e] : 0.f;
    double s = in ? sum_splits(e, (int)((long long)splits * sg / SG), (int)((long long)splits * (sg + 1) / SG)) : 0.0;
    s_part[sg][x] = s;
    __syncthreads();
    if (in && sg == 0) {
#pragma unroll
      for (int k = 1; k < SG; ++k) s += s_part[k][x];
      const float g = (float)s;
      grad[e] = g;
      if (W != nullptr) {
        const int r = (int)(e / ldp), c = (int)(e - (long long)r * ldp);
        if (c < cols) {
          grad_t[(long long)c * ldt + r] = g;
          if (r == rows - 1)
            for (int pad = rows; pad < ldt; ++pad) grad_t[(long long)c * ldt + pad] = 0.f;
        }
        sq[0] = (double)g * (double)g;
        sq[1] = (double)w * (double)w;
        most[0] = fabsf(g);
        most[1] = fabsf(w);
      }
    }
  }
  if (W == nullptr) return;
  // The sums, and in passing the maxima: a warp's go to shared memory before block_sums, whose barriers hand them to thread 0.
  __shared__ unsigned s_most[8][2];   // magnitudes: their order is that of their bits
  const auto block_totals = [&](uint2& top) {
    if (maxima) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(most[j]));
        if ((threadIdx.x & 31) == 0) s_most[threadIdx.x >> 5][j] = m;
      }
    }
    block_sums(sq, sh);
    top = make_uint2(0u, 0u);
    if (maxima && threadIdx.x == 0)
#pragma unroll
      for (int w = 0; w < 8; ++w) top = make_uint2(max(top.x, s_most[w][0]), max(top.y, s_most[w][1]));
  };
  uint2 top;
  block_totals(top);
  if (threadIdx.x == 0) {
    partial[3 * (size_t)blockIdx.x] = sq[0];
    partial[3 * (size_t)blockIdx.x + 1] = sq[1];
    if (maxima) reinterpret_cast<uint2*>(partial)[3 * (size_t)blockIdx.x + 2] = top;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sq[0] = sq[1] = 0.0;
  most[0] = most[1] = 0.f;
#pragma unroll 4
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    sq[0] += __ldcg(partial + 3 * (size_t)b);
    sq[1] += __ldcg(partial + 3 * (size_t)b + 1);
    if (!maxima) continue;
    const uint2 m = __ldcg(reinterpret_cast<const uint2*>(partial) + 3 * (size_t)b + 2);
    most[0] = fmaxf(most[0], __uint_as_float(m.x));
    most[1] = fmaxf(most[1], __uint_as_float(m.y));
  }
  block_totals(top);
  if (threadIdx.x == 0) {
    *ticket = 0;
    if (maxima) { ctl->g_max = __uint_as_float(top.x); ctl->w_max = __uint_as_float(top.y); }
    begin_one(ctl, sq[0], sq[1], shrink, growth, nullptr, status);
  }
}

// Search and move of a W block.  Along W - grad/t the pre-activation is H - D/t with D = P grad, so every candidate is
// scored from H, D, Z without another product:
//   hidden layer: sum_j = sum ( (z - f(h - d/t_j))^2 - (z - f(h))^2 )   (times nu/2 at decision time), kCand trials a sweep;
//                 one cooperative launch, k_search_w_hidden
//   last layer:   phi_L(t) - phi_L = -(1/t) <D, R> + (rho / 2t^2) ||D||^2 : two sums decide every trial, taken by the last
//                 block of k_score_w_out; k_move_w_out follows (ordinary launches: this chain runs beside the hidden layers')
// Then W <- W - grad/tau (and its transpose), H <- H - D/tau and, where Rn is given, the derivative of phi_l at the new
// H, which the gradient of Z_{l-1} starts from (formed here it costs one array less than in a sweep of its own).
struct SearchW {
  float4* H;
  const float4 *D, *Z, *U, *R;      // R: residual at the old H (last layer); U: last layer, for Rn
  float4* Rn;
  long long n4;
  float coef;                       // nu (hidden) or rho (last layer)
  float *W, *Wt;
  gtc::Image image, image_t;        // of W as the operand of P W and of S W^T
  const float* grad;
  int rows, cols, ldw, ldwt;
  SearchCtl* ctl;
  double* partial;                  // kCand (2) per block
  GridBar* bar;
  unsigned* ticket;
  int *status, *err;
  DecideArgs a;
  DecisionLog log;
};

template <bool OUT>
__device__ __forceinline__ void move_w(const SearchW& p, float step) {
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  if (step != 0.f) {
    __shared__ WeightTile turn;
    const int tiles = ((p.rows + 31) / 32) * ((p.cols + 31) / 32);
    const float bound = gtc::finite_bound(fmaf(step, __ldcg(&p.ctl->g_max), __ldcg(&p.ctl->w_max))), scale = gtc::scale_of(bound);   // |W - step grad| elementwise
    if (blockIdx.x == 0) {
      gtc::put_scales(p.image, p.cols, bound);
      gtc::put_scales(p.image_t, p.rows, bound);
    }
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      int marks = 0;
      weight_tile(tile, p.rows, p.cols, p.cols, turn, p.Wt, p.ldwt, p.image, p.image_t, scale, [&](int r, int c) {
        const long long e = (long long)r * p.ldw + c;
        const float w = fmaf(-p.grad[e], step, p.W[e]);
        p.W[e] = w;
        marks |= gtc::marks_for(w, scale);
        return w;
      });
      if (p.image.data != nullptr || p.image_t.data != nullptr) {
        marks = (__syncthreads_or(marks & gtc::kBelowPairs) ? gtc::kBelowPairs : 0) | (__syncthreads_or(marks & gtc::kWide) ? gtc::kWide : 0);
        if (threadIdx.x == 0) {   // a mark per tile, in both images: as many tiles in one as in the other
          if (p.image.data != nullptr) gtc::marks_of(p.image, p.cols)[tile] = marks;
          if (p.image_t.data != nullptr) gtc::marks_of(p.image_t, p.rows)[tile] = marks;
        }
      }
    }
  }
  if (step == 0.f && p.Rn == nullptr) return;
  for (long long i = first; i < p.n4; i += stride) {
    float4 h = p.H[i];
    if (step != 0.f) {
      h = vfma(-step, p.D[i], h);
      p.H[i] = h;
    }
    if (p.Rn != nullptr) p.Rn[i] = OUT ? resid_out(h, p.Z[i], p.U[i], p.coef) : resid_hidden(h, p.Z[i], p.coef);
  }
}

__global__ void __launch_bounds__(256, 4)
k_search_w_hidden(const SearchW p) {
  __shared__ double sh[kCand * 8], total[kCand];
  SearchCtl* const ctl = p.ctl;
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  const int gave_up = __ldcg(p.err), skipped = ctl->done;   // side by side: one latency
  if (gave_up != 0) return;         // see GridBar
  if (skipped) {                    // the same in every block
    if (first == 0) log_decision(p.log, 0, ctl);
  } else {
    bool open = true;
    while (open) {
      double s[kCand];
#pragma unroll
      for (int j = 0; j < kCand; ++j) s[j] = 0.0;
      float inv[kCand];
#pragma unroll
      for (int j = 0; j < kCand; ++j) inv[j] = __ldcg(&ctl->inv_cand[j]);
      for (long long i = first; i < p.n4; i += stride) {
        const float4 h4 = p.H[i], d4 = p.D[i], z4 = p.Z[i];
        const float h[4] = {h4.x, h4.y, h4.z, h4.w}, d[4] = {d4.x, d4.y, d4.z, d4.w}, z[4] = {z4.x, z4.y, z4.z, z4.w};
        float part[kCand];
#pragma unroll
        for (int j = 0; j < kCand; ++j) part[j] = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float pos = fmaxf(h[c], 0.f), neg = fmaxf(-h[c], 0.f);
          const float e2 = 2.f * (z[c] - pos);
#pragma unroll
          for (int j = 0; j < kCand; ++j) {
            const float df = relu_drop(d[c], inv[j], neg, pos);
            part[j] = fmaf(df, e2 + df, part[j]);   // e1^2 - e0^2 = (e1 - e0)(e1 + e0), e1 - e0 = df
          }
        }
#pragma unroll
        for (int j = 0; j < kCand; ++j) s[j] += (double)part[j];
      }
      block_sums(s, sh);
      if (threadIdx.x == 0)
#pragma unroll
        for (int j = 0; j < kCand; ++j) p.partial[(size_t)blockIdx.x * kCand + j] = s[j];
      const bool ok = grid_meet(p.bar, p.err, [&] {
        add_block_sums<kCand>(p.partial, (int)gridDim.x, total);
        if (threadIdx.x < 32 && !decide_one(ctl, total, 0.0, p.a, nullptr, p.status) && threadIdx.x == 0) log_decision(p.log, 0, ctl);
      });
      if (!ok) return;
      open = __ldcg(&ctl->done) == 0;
    }
  }
  move_w<false>(p, __ldcg(&ctl->inv_step));
}

__global__ void __launch_bounds__(256)
k_score_w_out(const SearchW p) {
  gtc::enter_kernel();
  __shared__ double sh[16], total[2];
  __shared__ int s_last;
  if (p.ctl->done) {                // skipped: the same in every block
    if (blockIdx.x == 0 && threadIdx.x == 0) log_decision(p.log, 0, p.ctl);
    return;
  }
  double s[2] = {0.0, 0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < p.n4; i += (long long)gridDim.x * blockDim.x) {
    const float4 d = p.D[i], r = p.R[i];
    s[0] += (double)(d.x * r.x + d.y * r.y + d.z * r.z + d.w * r.w);
    s[1] += (double)(d.x * d.x + d.y * d.y + d.z * d.z + d.w * d.w);
  }
  block_sums(s, sh);
  if (threadIdx.x == 0) {
    p.partial[(size_t)blockIdx.x * 2] = s[0];
    p.partial[(size_t)blockIdx.x * 2 + 1] = s[1];
    __threadfence();
    s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  add_block_sums<2>(p.partial, (int)gridDim.x, total);
  if (threadIdx.x >= 32) return;
  decide_one(p.ctl, total, 0.0, p.a, nullptr, p.status);
  if (threadIdx.x == 0) {
    *p.ticket = 0;
    log_decision(p.log, 0, p.ctl);
  }
}

__global__ void __launch_bounds__(256)
k_move_w_out(const SearchW p) {
  gtc::enter_kernel();
  move_w<true>(p, p.ctl->inv_step);
}

// The end of a pass: the pass counter of the log moves on, and with it the count of passes since H_1 was last formed afresh
// (*skip_h1 = 1 while H_1, which the W_1 update keeps equal to P_1 W_1 up to rounding, need not be).
__global__ void k_end_pass(int* __restrict__ pass, int* __restrict__ h1_age, int* __restrict__ skip_h1, int every) {
  gtc::enter_kernel();
  *pass += 1;
  const int age = *skip_h1 ? *h1_age + 1 : 0;   // the pass that has just ended formed H_1 unless *skip_h1 said not to
  *h1_age = age;
  *skip_h1 = age + 1 < every;
}

// Marks every entry of the current pass's slot as "not run".
__global__ void k_log_clear(int* __restrict__ trial_base, const int* __restrict__ pass, long long per_pass, int ring) {
  const long long at0 = (long long)(*pass % ring) * per_pass;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < per_pass;
       i += (long long)gridDim.x * blockDim.x)
    trial_base[at0 + i] = -3;
}

// ------------------------------------------------------------------------------------------
// Hidden Z blocks (Appendix A).  The gradient of psi_m with respect to Z_{l,m} is the rows V_m of
//   G = nu (Z_l - f(H_l)) + (A~ R') W_{l+1}^T ,
// R' the residual of layer l+1 at the new W.  k_zgrad_finish adds the first term to the product and forms, per
// community, { ||G||^2, ||Z_l||^2, <Z_l - f(H_l), G> }.  blocks[b] = {first row, one past the last, community, 0}: a
// block never crosses a community boundary and leaves the sums of its rows in partial[b*3 + ..]; the last block of a
// community to finish (tickets[m], left at zero) adds the community's blocks block_ptr[m] .. block_ptr[m+1]-1 up in a
// fixed order and starts its search.  A group of LPR lanes takes a row; row_max (may be NULL): the largest magnitude of every row of G.
// ------------------------------------------------------------------------------------------
// The sums t of row block `block` of community m, and what follows when it is the community's last to finish; the whole block.
__device__ __forceinline__ void close_zgrad(double (&t)[3], int block, int m, double* sh, double* partial, const int* __restrict__ block_ptr,
                                            unsigned* tickets, SearchCtl* ctl, double* __restrict__ sums, double shrink, double growth,
                                            int* n_active, int* status) {
  __shared__ int s_last;
  block_sums(t, sh);
  const int b0 = block_ptr[m], b1 = block_ptr[m + 1];
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < 3; ++j) partial[(size_t)block * 3 + j] = t[j];
    __threadfence();
    s_last = atomicAdd(tickets + m, 1u) == (unsigned)(b1 - b0) - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
#pragma unroll
  for (int j = 0; j < 3; ++j) t[j] = 0.0;
  for (int b = b0 + threadIdx.x; b < b1; b += blockDim.x)
#pragma unroll
    for (int j = 0; j < 3; ++j) t[j] += __ldcg(partial + (size_t)b * 3 + j);
  block_sums(t, sh);
  if (threadIdx.x == 0) {
    tickets[m] = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) sums[m * 3 + j] = t[j];
    begin_one(ctl + m, t[0], t[1], shrink, growth, n_active, status);
  }
}

template <int LPR>
__global__ void __launch_bounds__(256)
k_zgrad_finish(float4* __restrict__ G, const float4* __restrict__ Z, const float4* __restrict__ H, int ld4,
               const int4* __restrict__ blocks, float nu, double* partial, const int* __restrict__ block_ptr, unsigned* tickets,
               SearchCtl* ctl, double* __restrict__ sums, double shrink, double growth, int* n_active, int* status, float* __restrict__ row_max) {
  gtc::enter_kernel();
  __shared__ double sh[24];
  const int4 rb = blocks[blockIdx.x];
  double t[3] = {0.0, 0.0, 0.0};
  const int sub = threadIdx.x & (LPR - 1);
  for (int row = rb.x + (int)(threadIdx.x / LPR); __any_sync(0xffffffffu, row < rb.y); row += 256 / LPR) {
    const long long at = (long long)row * ld4;
    float big = 0.f;
    if (row < rb.y) {
#pragma unroll 2
      for (int f = sub; f < ld4; f += LPR) {
        const float4 z = Z[at + f], h = H[at + f];
        float4 g = G[at + f];
        const float ax = z.x - relu(h.x), ay = z.y - relu(h.y), az = z.z - relu(h.z), aw = z.w - relu(h.w);
        g.x = fmaf(nu, ax, g.x); g.y = fmaf(nu, ay, g.y); g.z = fmaf(nu, az, g.z); g.w = fmaf(nu, aw, g.w);
        G[at + f] = g;
        big = fmaxf(big, vabsmax(g));
        t[0] += (double)(g.x * g.x + g.y * g.y + g.z * g.z + g.w * g.w);
        t[1] += (double)(z.x * z.x + z.y * z.y + z.z * z.z + z.w * z.w);
        t[2] += (double)(ax * g.x + ay * g.y + az * g.z + aw * g.w);
      }
    }
    if (row_max != nullptr) {
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
      if (sub == 0 && row < rb.y) row_max[row] = big;
    }
  }
  close_zgrad(t, (int)blockIdx.x, rb.z, sh, partial, block_ptr, tickets, ctl, sums, shrink, growth, n_active, status);
}

// The same with both products beside it, for a narrow next layer: G[i] = S[i] W^T + nu (Z[i] - f(H[i])) and T[i] = G[i] W are rows of
// their own, so that G is written once and not read again (three launches and G through memory three times otherwise).  fp32 FMA.
// W^T lies in shared memory, 4 KV rows of ld4 float4 (those past the layer's width zero).  Eight lanes take R rows of G, so that a
// value of W serves R; shared memory is read 4 KV times per R float4 of G for each product, which with the registers of a row's S
// and T is what bounds it where HBM does not (see joins_products).  At KV = 12 these do not fit: 255 registers and 540 bytes of spills, on
// graphs of up to 4,096 rows only.
template <int KV, int R>
__global__ void __launch_bounds__(256 / R)
k_zgrad_products(float4* __restrict__ G, const float4* __restrict__ Z, const float4* __restrict__ H, const float4* __restrict__ S,
                 const float4* __restrict__ Wt, float4* __restrict__ T, int ld4, int next_cols, const int4* __restrict__ blocks,
                 int n_blocks, float nu, double* partial, const int* __restrict__ block_ptr, unsigned* tickets, SearchCtl* ctl,
                 double* __restrict__ sums, double shrink, double growth, int* n_active, int* status) {
  gtc::enter_kernel();
  extern __shared__ float4 s_wt[];
  __shared__ double sh[24];
  int4 rb = blocks[blockIdx.x];   // beside the first loads of W
  for (int i = threadIdx.x; i < 4 * KV * ld4; i += blockDim.x) s_wt[i] = i < next_cols * ld4 ? Wt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int sub = threadIdx.x & 7, group = threadIdx.x >> 3, next4 = (next_cols + 3) / 4;
  for (int blk = blockIdx.x; blk < n_blocks; blk += gridDim.x) {
    if (blk != (int)blockIdx.x) rb = blocks[blk];
    double t[3] = {0.0, 0.0, 0.0};
    const int row = rb.x + R * group;   // the first of this group's rows: a block has R for each of its groups
    bool in[R];
    float s[R][4 * KV], out[R][4 * KV];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      in[j] = row + j < rb.y;
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const float4 v = in[j] && k < next4 ? S[(long long)(row + j) * next4 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
        s[j][4 * k] = v.x; s[j][4 * k + 1] = v.y; s[j][4 * k + 2] = v.z; s[j][4 * k + 3] = v.w;
        out[j][4 * k] = out[j][4 * k + 1] = out[j][4 * k + 2] = out[j][4 * k + 3] = 0.f;
      }
    }
    for (int f = sub; f < ld4; f += 8) {
      float4 z[R], h[R], g[R];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        z[j] = h[j] = g[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in[j]) { z[j] = Z[(long long)(row + j) * ld4 + f]; h[j] = H[(long long)(row + j) * ld4 + f]; }
      }
#pragma unroll
      for (int k = 0; k < 4 * KV; ++k) {
        const float4 w = s_wt[k * ld4 + f];
#pragma unroll
        for (int j = 0; j < R; ++j) g[j] = vfma(s[j][k], w, g[j]);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const float ax = z[j].x - relu(h[j].x), ay = z[j].y - relu(h[j].y), az = z[j].z - relu(h[j].z), aw = z[j].w - relu(h[j].w);
        g[j].x = fmaf(nu, ax, g[j].x); g[j].y = fmaf(nu, ay, g[j].y); g[j].z = fmaf(nu, az, g[j].z); g[j].w = fmaf(nu, aw, g[j].w);
        if (in[j]) G[(long long)(row + j) * ld4 + f] = g[j];
        t[0] += (double)(g[j].x * g[j].x + g[j].y * g[j].y + g[j].z * g[j].z + g[j].w * g[j].w);
        t[1] += (double)(z[j].x * z[j].x + z[j].y * z[j].y + z[j].z * z[j].z + z[j].w * z[j].w);
        t[2] += (double)(ax * g[j].x + ay * g[j].y + az * g[j].z + aw * g[j].w);
      }
#pragma unroll
      for (int k = 0; k < 4 * KV; ++k) {
        const float4 w = s_wt[k * ld4 + f];
#pragma unroll
        for (int j = 0; j < R; ++j)
          out[j][k] = fmaf(g[j].w, w.w, fmaf(g[j].z, w.z, fmaf(g[j].y, w.y, fmaf(g[j].x, w.x, out[j][k]))));
      }
    }
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
      for (int k = 0; k < 4 * KV; ++k)
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) out[j][k] += __shfl_xor_sync(0xffffffffu, out[j][k], o);
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
      for (int k = 0; k < KV; ++k)
        if (in[j] && k < next4 && sub == ((j * KV + k) & 7))
          T[(long long)(row + j) * next4 + k] = make_float4(out[j][4 * k], out[j][4 * k + 1], out[j][4 * k + 2], out[j][4 * k + 3]);
    close_zgrad(t, blk, rb.z, sh, partial, block_ptr, tickets, ctl, sums, shrink, growth, n_active, status);
    __syncthreads();   // its shared memory is free again
  }
}

// Warp-wide sums of 4 per-lane values with 6 shuffles: lane 8*j ends up holding the total of value j.
__device__ __forceinline__ float warp_sum4(float v0, float v1, float v2, float v3, int lane) {
  const bool up16 = lane & 16, up8 = lane & 8;
  const float r0 = __shfl_xor_sync(0xffffffffu, up16 ? v0 : v2, 16);
  const float r1 = __shfl_xor_sync(0xffffffffu, up16 ? v1 : v3, 16);
  const float a = (up16 ? v2 : v0) + r0, b = (up16 ? v3 : v1) + r1;
  float c = (up8 ? b : a) + __shfl_xor_sync(0xffffffffu, up8 ? a : b, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

// Scoring of the theta candidates of every community in one sweep over the rows.
// With T = G W_{l+1}, the move of community m changes the pre-activation of row i by
//   -K_m[i] / theta_m ,  K_m[i] = sum over j in V_m of A~_ij T_j  (row i of A~_{comm(i),m} T_m),
// which is non-zero on V_m and its first-order neighbour rows only.  A warp owns row i and walks
// its stored entries once; col_comm gives the community of every entry, entries of one community
// are contiguous (ascending columns), and at every change of community the finished K_m[i] is scored:
//   per community, sum_c (z - f(h - k/t_j))^2 - (z - f(h))^2 for j < kCand
//                                        (a candidate costs two instructions per element, and a search
//                                        that needs more trials than one sweep scores is served by a
//                                        further sweep; two or three per sweep gained 8 % of the first
//                                        sweep at most and brought later ones back)
// (Layer l+1 = L is linear and has a search of its own, k_search_z_out.)
// Sums are kept per warp in shared memory (no atomics on the hot path) and leave the kernel per chunk of
// units (see the scheduling note in the kernel).  V = float4 columns per lane (width <= 128 V).
// Persistent grid.
//
// Rows longer than `long_len` come as `n_items` items {row, first entry, one past the last, split}
// (see k_spmm_wide): an item of whole community segments (split < 0) is scored like a short row; an
// item that is one piece of a segment too long for one warp only leaves its part of K_m[i],
// unscaled, in `scratch` (one padded row per item), and k_close_z scores the sum of the pieces.

// 2 (z - f(h)): twice the row's current error, formed once per row and reused by every segment.
__device__ __forceinline__ float4 twice_error(const float4& h, const float4& z) {
  return make_float4(2.f * (z.x - relu(h.x)), 2.f * (z.y - relu(h.y)), 2.f * (z.z - relu(h.z)), 2.f * (z.w - relu(h.w)));
}

// Scores one finished K_m[i] (k, still without the factor di) against the row's a, b:
// a = h and b = twice_error(h, z).  The kCand sums go to `slots`:
// add: added to what is there (the slots belong to this warp), else stored.
__device__ __forceinline__ void put_sum(double* dst, float r, bool add) { *dst = add ? *dst + (double)r : (double)r; }
template <int V>
__device__ __forceinline__ void score_segment(const float4 (&k)[V], float di, const float4 (&a)[V],
                                              const float4 (&b)[V], const float* inv_cand, int lane, double* slots,
                                              bool add) {
  static_assert(kCand == 4, "warp_sum4 and the float4 of a community's candidates hold four");
  float inv[kCand], part[kCand];
#pragma unroll
  for (int j = 0; j < kCand; ++j) { inv[j] = di * inv_cand[j]; part[j] = 0.f; }   // K_m[i] = di * k
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const float kk[4] = {k[v].x, k[v].y, k[v].z, k[v].w};
    const float hh[4] = {a[v].x, a[v].y, a[v].z, a[v].w};
    const float ee[4] = {b[v].x, b[v].y, b[v].z, b[v].w};   // 2 (z - f(h)), see twice_error
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float pos = fmaxf(hh[c], 0.f), neg = fmaxf(-hh[c], 0.f);
#pragma unroll
      for (int j = 0; j < kCand; ++j) {
        const float df = relu_drop(kk[c], inv[j], neg, pos);
        part[j] = fmaf(df, ee[c] + df, part[j]);   // e1^2 - e0^2 = df (2 e0 + df)
      }
    }
  }
  const float r = warp_sum4(part[0], part[1], part[2], part[3], lane);
  if ((lane & 7) == 0) put_sum(slots + (lane >> 3), r, add);
}

// What the search of a hidden layer's Z blocks needs beside the scoring kernel's own operands.
struct SearchZ {
  SearchCtl* ctl;                    // one per community
  int n_comm;
  double* chunk_part;                // [chunk][community][sums] of a sweep
  int* chunk_counter;                // hands the chunks out; left at zero
  double* group_part;                // [group of chunks][community][sums], used when n_groups > 0
  int n_groups, per_group;
  const int4* split;                 // segments scored in pieces: {row, community, first item, number of items}
  int n_split;
  double* split_scores;
  const int *split_order, *split_ptr;   // their order by community
  const double* own;                 // [community][3] from k_zgrad_finish; [2] = <Z - f(H), G>
  int *n_active, *status, *err;
  GridBar* bar;
  DecideArgs a;
  DecisionLog log;
  float4* Z;                         // the block that moves, its gradient, their width, community of every row
  const float4* G;
  int ldz4;
  const int* row_comm;
};

// Closes a sweep.  Segments that were scored in pieces: K_m[i] = sum of the pieces (item order), then scored like any
// other, one warp each.  With many chunks their sums are first added group by group, in chunk order.  Then one warp per
// community adds up its groups (or chunks; lane-strided, then the shuffle tree) and its split segments in table order,
// and takes the decision.  No sum depends on which warp scored which chunk.
template <int V>
__device__ __forceinline__ bool close_sweep(const SearchZ& p, int n_chunks, const float* __restrict__ dinv, const float4* scratch,
                                            const float4* __restrict__ Hn, const float4* __restrict__ Zn, int ld4) {
  constexpr int PER = kCand;
  const int lane = threadIdx.x & 31;
  const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), n_warps = (int)((gridDim.x * blockDim.x) >> 5);
  const auto nothing = [] {};
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.chunk_counter = 0;
  if (p.n_split > 0 || p.n_groups > 0) {
    for (int s = gwarp; s < p.n_split; s += n_warps) {
      const int4 sp = p.split[s];
      if (p.ctl[sp.y].done) continue;
      float4 a[V], b[V], k[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int f = lane + 32 * v;
        a[v] = b[v] = k[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (f < ld4) {
          a[v] = Hn[(long long)sp.x * ld4 + f];
          b[v] = twice_error(a[v], Zn[(long long)sp.x * ld4 + f]);
          for (int q = 0; q < sp.w; ++q) k[v] = vadd(k[v], __ldcg(scratch + (long long)(sp.z + q) * ld4 + f));
        }
      }
      score_segment<V>(k, dinv[sp.x], a, b, p.ctl[sp.y].inv_cand, lane, p.split_scores + (size_t)s * PER, false);
    }
    const int width = p.n_comm * PER;
    for (int g = blockIdx.x; g < p.n_groups; g += gridDim.x) {
      const int c1 = min(n_chunks, (g + 1) * p.per_group);
      for (int v = threadIdx.x; v < width; v += blockDim.x) {
        double s = 0.0;
#pragma unroll 8
        for (int ch = g * p.per_group; ch < c1; ++ch) s += __ldcg(p.chunk_part + (size_t)ch * width + v);
        p.group_part[(size_t)g * width + v] = s;
      }
    }
    if (!grid_meet(p.bar, p.err, nothing)) return false;
  }
  const double* const parts = p.n_groups > 0 ? p.group_part : p.chunk_part;
  const int n_parts = p.n_groups > 0 ? p.n_groups : n_chunks;
  for (int i = gwarp; i < p.n_comm; i += n_warps) {
    SearchCtl* c = p.ctl + i;
    if (c->done) continue;
    double s[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) s[j] = 0.0;
    for (int b = lane; b < n_parts; b += 32)
#pragma unroll
      for (int j = 0; j < PER; ++j) s[j] += __ldcg(parts + ((size_t)b * p.n_comm + i) * PER + j);
    for (int k = p.split_ptr[i] + lane; k < p.split_ptr[i + 1]; k += 32) {
      const size_t at = (size_t)p.split_order[k] * PER;
#pragma unroll
      for (int j = 0; j < PER; ++j) s[j] += __ldcg(p.split_scores + at + j);
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) s[j] = warp_sum(s[j]);
    decide_one(c, s, p.own[i * 3 + 2], p.a, p.n_active, p.status);
  }
  return grid_meet(p.bar, p.err, nothing);
}

// After the last sweep: the decisions go to the log and every block moves, Z_l[i,:] <- Z_l[i,:] - G[i,:] / theta_{comm(i)} (Eq. 10).
__device__ __forceinline__ void move_blocks(const SearchZ& p, long long n) {
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < p.n_comm; i += stride) log_decision(p.log, (int)i, p.ctl + i);
  // four elements per thread in flight: the kernel holds few warps (its scoring loop takes the registers)
  const long long total = n * p.ldz4;   // below 2^32
  for (long long e0 = first; e0 < total; e0 += 4 * stride) {
    float s[4];
    float4 g[4], z[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long e = e0 + k * stride;
      s[k] = 0.f;
      if (e < total) {
        s[k] = p.ctl[p.row_comm[(unsigned)e / (unsigned)p.ldz4]].inv_step;
        g[k] = __ldcs(p.G + e);
        z[k] = p.Z[e];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (s[k] != 0.f) p.Z[e0 + k * stride] = vfma(-s[k], g[k], z[k]);
  }
}

// One sweep over all chunks by the warps of the grid.  Dynamic shared memory: per warp the row's a, b (2 V float4 per
// lane; parked there during the walk so that the registers hold gathered rows instead), the candidates of every community
// (one float4; negative when its search is closed), then the per-warp sums; the last two only with use_smem.
template <int V, int UN>
__device__ __forceinline__ void score_sweep(const int* __restrict__ row_ptr, const int* __restrict__ col,
          const unsigned short* __restrict__ col_comm, const float* __restrict__ dinv,
          const float4* __restrict__ T, const float4* __restrict__ Hn, const float4* __restrict__ Zn, int ld4, const SearchCtl* ctl, int n_comm, double* chunk_part, int use_smem,
          const int* __restrict__ chunk_ptr, int n_chunks, int* chunk_counter,
          const int4* __restrict__ items, int n_items, int long_len, float4* scratch) {
  constexpr int PER = kCand;
  extern __shared__ float4 s_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int warps_per_block = blockDim.x >> 5;
  float4* row_ab = s_raw + (size_t)warp * (2 * V * 32) + lane;
  float4* const s_cand = s_raw + (size_t)warps_per_block * (2 * V * 32);
  double* s_acc = reinterpret_cast<double*>(s_cand + n_comm);
  double* mine = nullptr;   // the sums of the chunk in hand, [community][PER]
  if (use_smem) {
    for (int i = threadIdx.x; i < warps_per_block * n_comm * PER; i += blockDim.x) s_acc[i] = 0.0;
    mine = s_acc + (size_t)warp * n_comm * PER;
    for (int m = threadIdx.x; m < n_comm; m += blockDim.x) {   // written by other blocks in a sweep after the first: not through L1
      const SearchCtl* c = ctl + m;
      s_cand[m] = __ldcg(&c->done) ? make_float4(-1.f, 0.f, 0.f, 0.f)
                                   : make_float4(__ldcg(c->inv_cand), __ldcg(c->inv_cand + 1), __ldcg(c->inv_cand + 2), __ldcg(c->inv_cand + 3));
    }
  }
  __syncthreads();
  const float4* __restrict__ T_lane = T + lane;   // rows of T are addressed by 32-bit float4 offsets (n * ld4 < 2^32)
  bool in_row[V];
#pragma unroll
  for (int v = 0; v < V; ++v) in_row[v] = lane + 32 * v < ld4;
  // Units (items first, then rows) come in chunks of about equally many stored entries (chunk_ptr, built
  // on the host).  Chunks are handed out from a global counter (`chunk_counter`, zero at launch): row
  // lengths follow a power law and the time a chunk takes depends on what its rows find in L2, so any
  // static deal leaves most warps waiting for the unlucky ones.  A chunk is scored by one warp, units in
  // order, and its sums go to chunk_part[chunk][community][PER]; they are added up in chunk order
  // afterwards (close_sweep), so no sum depends on which warp took which chunk.
  // With room in shared memory the chunk's sums are kept there and copied out at the end of the chunk;
  // otherwise (too many communities) the warp adds into the chunk's slice of chunk_part directly.
  for (;;) {
    int ch = 0;
    if (lane == 0) ch = atomicAdd(chunk_counter, 1);
    ch = __shfl_sync(0xffffffffu, ch, 0);
    if (ch >= n_chunks) break;
    double* const out_part = chunk_part + (size_t)ch * n_comm * PER;
    if (!use_smem) {
      for (int i = lane; i < n_comm * PER; i += 32) out_part[i] = 0.0;
      mine = out_part;
      __syncwarp();
    }
    const int chunk_end = chunk_ptr[ch + 1];
  for (int unit_base = chunk_ptr[ch]; unit_base < chunk_end; unit_base += 4) {
    const int unit_end = min(chunk_end, unit_base + 4);
    // lanes 0..3 fetch the descriptions of the four units together (one load latency, not four)
    int4 my_unit = make_int4(0, 0, 0, -1);   // row, first entry, one past the last, split (>= 0: a piece)
    if (lane < 4 && unit_base + lane < unit_end) {
      const int u = unit_base + lane;
      if (u < n_items) my_unit = items[u];
      else {
        const int r = u - n_items;
        my_unit = make_int4(r, row_ptr[r], row_ptr[r + 1], -1);
        if (my_unit.z - my_unit.y > long_len) my_unit.z = my_unit.y;   // walked as items
      }
    }
    // column and community of a unit's first chunk are fetched while the unit before it is walked
    int c_first = 0, m_first = -1;
    {
      const int s0 = __shfl_sync(0xffffffffu, my_unit.y, 0), e0 = __shfl_sync(0xffffffffu, my_unit.z, 0);
      if (s0 + lane < e0) { c_first = col[s0 + lane]; m_first = col_comm[s0 + lane]; }
    }
  for (int unit = unit_base; unit < unit_end; ++unit) {
    const int q = unit - unit_base;
    const int row = __shfl_sync(0xffffffffu, my_unit.x, q);
    const int rs = __shfl_sync(0xffffffffu, my_unit.y, q), re = __shfl_sync(0xffffffffu, my_unit.z, q);
    const bool piece = __shfl_sync(0xffffffffu, my_unit.w, q) >= 0;
    int c_next = c_first, m_next = m_first;
    {
      const int s1 = __shfl_sync(0xffffffffu, my_unit.y, (q + 1) & 3), e1 = __shfl_sync(0xffffffffu, my_unit.z, (q + 1) & 3);
      m_first = -1;
      if (q + 1 < unit_end - unit_base && s1 + lane < e1) { c_first = col[s1 + lane]; m_first = col_comm[s1 + lane]; }
    }
    if (rs >= re) continue;
    __syncwarp();          // the previous unit's last segment has been scored
#pragma unroll
    for (int v = 0; v < V; ++v) {   // a = h, b = 2 (z - f(h))
      const int f = lane + 32 * v;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (f < ld4 && !piece) {
        { a = Hn[(long long)row * ld4 + f]; b = twice_error(a, Zn[(long long)row * ld4 + f]); }
      }
      row_ab[32 * v] = a;
      row_ab[32 * (V + v)] = b;
    }
    const float di = dinv[row];
    float4 k[V];
#pragma unroll
    for (int v = 0; v < V; ++v) k[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    int cur = -1;          // community of the segment being accumulated
    bool cur_on = false;   // its search is still running

    auto finish_segment = [&]() {
      if (!cur_on) return;
      if (piece) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int f = lane + 32 * v;
          if (f < ld4) scratch[(long long)unit * ld4 + f] = k[v];
        }
        return;
      }
      float4 a[V], b[V];   // each lane reads back what it stored itself
#pragma unroll
      for (int v = 0; v < V; ++v) {
        a[v] = row_ab[32 * v];
        b[v] = row_ab[32 * (V + v)];
      }
      score_segment<V>(k, di, a, b, use_smem ? reinterpret_cast<const float*>(s_cand + cur) : ctl[cur].inv_cand, lane,
                                mine + cur * PER, true);
    };

    // column and community of a chunk are fetched while the chunk before it is walked; the two
    // loads that depend on them (weight, search state) are issued together, not one after the other
    for (int base = rs; base < re; base += 32) {
      const int idx = base + lane;
      const bool valid = idx < re;
      const int c = c_next, m = m_next;
      if (idx + 32 < re) { c_next = col[idx + 32]; m_next = col_comm[idx + 32]; }
      else m_next = -1;
      unsigned off = 0u;      // first float4 of the entry's row of T; lanes past the row's end hold (row 0, weight 0)
      float w = 0.f;
      bool live = false;      // the entry's community is still searching: its row of T is gathered
      if (valid) {
        const float wc = dinv[c];
        live = use_smem ? s_cand[m].x >= 0.f : __ldcg(&ctl[m].done) == 0;
        if (live) { w = wc; off = (unsigned)c * (unsigned)ld4; }
      }
      // entries of one community are contiguous: bit t of `chg` says that entry t opens a new
      // segment, bit t of `on` that its row is gathered; both are the same in every lane, so the
      // walk below needs the community of an entry only where a segment starts
      int mprev = __shfl_up_sync(0xffffffffu, m, 1);
      if (lane == 0) mprev = cur;
      unsigned chg = __ballot_sync(0xffffffffu, valid && m != mprev);
      unsigned on = __ballot_sync(0xffffffffu, live);
      const int cnt = min(32, re - base);
      if (on == 0u) {   // nothing to gather in this chunk (the usual case in a sweep after the first)
        if (chg != 0u) {   // an open segment ends at the chunk's first entry; a later one starts from scratch
          finish_segment();
          cur = __shfl_sync(0xffffffffu, m, cnt - 1);
          cur_on = false;
        }
        continue;
      }
      for (int t = 0; t < cnt; t += UN, chg >>= UN, on >>= UN) {
        unsigned oj[UN];
        float wj[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          oj[u] = __shfl_sync(0xffffffffu, off, t + u);
          wj[u] = __shfl_sync(0xffffffffu, w, t + u);
        }
        float4 xv[UN][V];   // set and read under the same condition (entry gathered, column inside the row)
#pragma unroll
        for (int u = 0; u < UN; ++u)
#pragma unroll
          for (int v = 0; v < V; ++v)
            if (((on >> u) & 1u) && in_row[v]) xv[u][v] = __ldg(T_lane + oj[u] + 32 * v);
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          if ((chg >> u) & 1u) {                          // warp-uniform
            finish_segment();
            cur = __shfl_sync(0xffffffffu, m, t + u);
            cur_on = (on >> u) & 1u;
#pragma unroll
            for (int v = 0; v < V; ++v) k[v] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int v = 0; v < V; ++v)
            if (((on >> u) & 1u) && in_row[v]) {
              k[v].x = fmaf(wj[u], xv[u][v].x, k[v].x); k[v].y = fmaf(wj[u], xv[u][v].y, k[v].y);
              k[v].z = fmaf(wj[u], xv[u][v].z, k[v].z); k[v].w = fmaf(wj[u], xv[u][v].w, k[v].w);
            }
        }
      }
    }
    finish_segment();
  }
  }
    __syncwarp();
    if (use_smem)
      for (int i = lane; i < n_comm * PER; i += 32) { out_part[i] = mine[i]; mine[i] = 0.0; }
    __syncwarp();
  }
}

template <int V, int UN>
__global__ void __launch_bounds__(256, (V <= 1 ? 4 : V <= 2 ? 3 : 1))
k_score_z(const int* __restrict__ row_ptr, const int* __restrict__ col,
          const unsigned short* __restrict__ col_comm, const float* __restrict__ dinv,
          const float4* __restrict__ T, const float4* __restrict__ Hn, const float4* __restrict__ Zn, int ld4, const SearchCtl* __restrict__ ctl, int n_comm,
          double* __restrict__ chunk_part, const int* __restrict__ n_active, int use_smem,
          const int* __restrict__ chunk_ptr, int n_chunks, int* __restrict__ chunk_counter,
          const int4* __restrict__ items, int n_items, int long_len, float4* __restrict__ scratch) {
  if (*n_active <= 0) return;
  score_sweep<V, UN>(row_ptr, col, col_comm, dinv, T, Hn, Zn, ld4, ctl, n_comm, chunk_part, use_smem, chunk_ptr, n_chunks,
                              chunk_counter, items, n_items, long_len, scratch);
}

// The rest of the search, cooperative: closes the sweep that k_score_z has just made, makes and
// closes further ones while a community is still searching, and moves the blocks.  The first sweep has a
// kernel of its own because, compiled together with this one, its walk spills registers (2.4 M rows x 256: 14.9 against 13.6 ms).
// The searches of a launch start together, so the sweep that scores the last of max_trials is the last one: *n_active alone
// would not end the loop where a launch before this one gave up and left it too high.
template <int V, int UN>
__global__ void __launch_bounds__(256, (V <= 2 ? 3 : 1))
k_close_z(const int* __restrict__ row_ptr, const int* __restrict__ col,
          const unsigned short* __restrict__ col_comm, const float* __restrict__ dinv,
          const float4* __restrict__ T, const float4* __restrict__ Hn, const float4* __restrict__ Zn, int ld4, int n, int use_smem, const int* __restrict__ chunk_ptr, int n_chunks,
          const int4* __restrict__ items, int n_items, int long_len, float4* scratch, const SearchZ sz) {
  const int gave_up = __ldcg(sz.err), active = __ldcg(sz.n_active);   // side by side: one latency
  if (gave_up != 0) return;   // see GridBar
  if (active > 0) {
    for (int scored = sz.a.cand;; scored += sz.a.cand) {
      if (!close_sweep<V>(sz, n_chunks, dinv, scratch, Hn, Zn, ld4)) return;
      if (__ldcg(sz.n_active) <= 0 || scored >= sz.a.max_trials) break;   // *n_active changes only between the meetings of close_sweep
      score_sweep<V, UN>(row_ptr, col, col_comm, dinv, T, Hn, Zn, ld4, sz.ctl, sz.n_comm, sz.chunk_part, use_smem, chunk_ptr,
                                  n_chunks, sz.chunk_counter, items, n_items, long_len, scratch);
      if (!grid_meet(sz.bar, sz.err, [] {})) return;
    }
  }
  move_blocks(sz, n);
}

// ------------------------------------------------------------------------------------------
// The search of the last hidden layer (layer l+1 = L is linear): along Z_{l,m} - G_m/theta the objective changes by
//   -(1/theta) sum_i <K_m[i], R'_i> + (rho / 2 theta^2) sum_i ||K_m[i]||^2   plus the block's own quadratic term,
// so two sums decide every trial.  The first needs no walk over the graph: A~ is symmetric, hence
//   sum_i <K_m[i], R'_i> = sum_{j in V_m} <T_j, (A~ R')_j>,  and A~ R' = S has just been formed for the gradient.
// The second is a sum over the segments (row i, community m) of the graph, taken community by community (tables of
// build_segment_tables): the rows of T that a community's segments gather are the community's own block of T, a few MB that
// stay in L2, the segments of a chunk have one length, so the lanes of a warp never wait for each other, and a chunk
// belongs to one community, so that its sum lives in a register.
// (Walking the rows instead, with a ballot per group of entries to find the segments and a shared-memory slot per
// community: 45 us at 20 k rows x 3 classes, 146 us at 169 k x 40, 4.6 ms at 2.45 M x 47; this form: 21 us, 99 us, 3.8 ms.)
// CL lanes hold a row of T (ld4 <= CL float4), 32 / CL segments at a time per warp; segments of `share_from` entries or more
// are shared by all lanes of the warp, entry e going to set e mod (32 / CL).  The warp that finishes a community's last slot adds
// its slots up in slot order and takes the decision.  At the 80 registers of three blocks per SM every instantiation spills
// (100 to 332 bytes of stores); two blocks, and the decision as a function of its own, have not been measured.
// ------------------------------------------------------------------------------------------
struct SegRef {
  int begin;
  float dinv;
};
struct SegChunk {
  int first, count, length, comm, slot;   // see build_segment_tables
};
struct SearchOut {
  const SegRef* segs;
  const SegChunk* chunks;
  int n_chunks;
  int* chunk_counter;
  const int* slot_ptr;        // [n_comm + 1]
  double* slots;              // [slot][2]: sum of <T, S>, sum of ||K||^2
  int *comm_done, *split_done;   // finished slots of a community, finished pieces of a split segment; left at zero
  const int4 *items, *split;
  SearchCtl* ctl;
  const double* own;          // [community][3] from k_zgrad_finish; [2] = <Z - f(H), G>
  int *n_active, *status;
  int share_from;             // segments of this length or more are shared by all lanes of a warp
  DecideArgs a;
};

// dot and square sums of the float4 a lane holds
__device__ __forceinline__ float dot4(const float4& a, const float4& b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }

// `count` segments of length LEN <= 3.  The lanes fetch the entries of 32 segments, one segment each (columns of the
// next 32 while these are gathered), and hand them to the groups by shuffles; UN segments per group in flight.
template <int CL, int LEN, int UN>
__device__ __forceinline__ double short_segments(const SegRef* __restrict__ segs, int count, const int* __restrict__ col,
                                                 const float* __restrict__ dinv, const float4* __restrict__ T, int ld4, int lane) {
  constexpr int GROUPS = 32 / CL;
  const int grp = lane / CL, cl = lane & (CL - 1);
  const float4* __restrict__ T_lane = T + min(cl, ld4 - 1);
  double acc = 0.0;
  SegRef next{0, 0.f};
  if (lane < count) next = segs[lane];
  int c_next[LEN];
#pragma unroll
  for (int e = 0; e < LEN; ++e) c_next[e] = lane < count ? col[next.begin + e] : 0;
  for (int b = 0; b < count; b += 32) {
    const float di = next.dinv;
    int c[LEN];
    float w[LEN];
#pragma unroll
    for (int e = 0; e < LEN; ++e) { c[e] = c_next[e]; w[e] = dinv[c[e]]; }   // past the last segment: column 0, factor 0
    next.dinv = 0.f;
    const bool more = b + 32 + lane < count;
    if (more) next = segs[b + 32 + lane];
#pragma unroll
    for (int e = 0; e < LEN; ++e) c_next[e] = more ? col[next.begin + e] : 0;
    const int nb = min(32, count - b);
    for (int t = 0; t * GROUPS < nb; t += UN) {
      float part = 0.f;
      float4 x[UN][LEN];
      float ww[UN][LEN], dd[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int src = ((t + u) * GROUPS + grp) & 31;
        dd[u] = __shfl_sync(0xffffffffu, di, src);
        if ((t + u) * GROUPS >= 32) dd[u] = 0.f;
#pragma unroll
        for (int e = 0; e < LEN; ++e) {
          const int r = __shfl_sync(0xffffffffu, c[e], src);
          ww[u][e] = __shfl_sync(0xffffffffu, w[e], src);
          x[u][e] = __ldg(T_lane + (unsigned)r * (unsigned)ld4);   // n * ld4 < 2^32; lanes past the row read its last column
        }
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        float4 k = vscale(ww[u][0], x[u][0]);
#pragma unroll
        for (int e = 1; e < LEN; ++e) k = vfma(ww[u][e], x[u][e], k);
        k = vscale(dd[u], k);
        part += dot4(k, k);
      }
      if (cl < ld4) acc += (double)part;
    }
  }
  return acc;
}

// `count` segments of one length, a group of CL >= 8 lanes each: the group's lanes fetch CL entries at a time, columns two
// steps ahead and weights one (across segments too), and hand them round by shuffles.
template <int CL, int UN>
__device__ __forceinline__ double group_segments(const SegRef* __restrict__ segs, int count, int len, const int* __restrict__ col,
                                                 const float* __restrict__ dinv, const float4* __restrict__ T, int ld4, int lane) {
  constexpr int GROUPS = 32 / CL;
  const int grp = lane / CL, cl = lane & (CL - 1);
  const bool in_row = cl < ld4;
  const float4* __restrict__ T_lane = T + cl;
  double acc = 0.0;
  int f_k = grp, f_o = cl, f_begin = grp < count ? segs[grp].begin : 0, f_next = grp + GROUPS < count ? segs[grp + GROUPS].begin : 0;
  auto fetch = [&]() {   // the next column of this lane; -1 past a segment's end
    const int c = f_k < count && f_o < len ? col[f_begin + f_o] : -1;
    f_o += CL;
    if (f_o - cl >= len) {   // the same in all groups
      f_o = cl;
      f_k += GROUPS;
      f_begin = f_next;
      if (f_k + GROUPS < count) f_next = segs[f_k + GROUPS].begin;
    }
    return c;
  };
  int c_n = fetch(), c_n2 = fetch();
  float w_n = c_n >= 0 ? dinv[c_n] : 0.f;
  for (int k0 = 0; k0 < count; k0 += GROUPS) {
    float4 k;
    vzero(k);
    for (int o = 0; o < len; o += CL) {
      const int c = max(c_n, 0);
      const float w = w_n;
      c_n = c_n2;
      w_n = c_n >= 0 ? dinv[c_n] : 0.f;
      c_n2 = fetch();
      const int cnt = min(CL, len - o);
      for (int t = 0; t < cnt; t += UN) {
        int r[UN];
        float ww[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          r[u] = __shfl_sync(0xffffffffu, c, t + u, CL);
          ww[u] = __shfl_sync(0xffffffffu, w, t + u, CL);
        }
        if (in_row) {
          float4 x[UN];
#pragma unroll
          for (int u = 0; u < UN; ++u) x[u] = __ldg(T_lane + (unsigned)r[u] * (unsigned)ld4);   // n * ld4 < 2^32
#pragma unroll
          for (int u = 0; u < UN; ++u) k = vfma(ww[u], x[u], k);
        }
      }
    }
    if (k0 + grp < count) {
      k = vscale(segs[k0 + grp].dinv, k);
      acc += (double)dot4(k, k);
    }
  }
  return acc;
}

// K_m[i] / dinv_i of one run of entries [b, e), entry b + set, b + set + sets, .. of it
template <int UN>
__device__ __forceinline__ float4 walk_run(int b, int e, int set, int sets, const int* __restrict__ col, const float* __restrict__ dinv,
                                           const float4* __restrict__ T, int ld4, int cl) {
  float4 k;
  vzero(k);
  int c[UN];
#pragma unroll
  for (int u = 0; u < UN; ++u) c[u] = b + set + u * sets < e ? col[b + set + u * sets] : -1;
  for (int p = b + set; p < e; p += UN * sets) {
    float w[UN];
    int r[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) { r[u] = c[u]; w[u] = r[u] >= 0 ? dinv[r[u]] : 0.f; }
    const int q = p + UN * sets;
#pragma unroll
    for (int u = 0; u < UN; ++u) c[u] = q + u * sets < e ? col[q + u * sets] : -1;
    if (cl < ld4) {
      float4 x[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u)
        if (r[u] >= 0) x[u] = __ldg(T + (long long)r[u] * ld4 + cl);
#pragma unroll
      for (int u = 0; u < UN; ++u)
        if (r[u] >= 0) k = vfma(w[u], x[u], k);
    }
  }
  return k;
}
// sum over the sets of a warp that share a run
template <int CL>
__device__ __forceinline__ float4 add_sets(float4 k) {
#pragma unroll
  for (int o = CL; o < 32; o <<= 1) k = vadd(k, vxor(0xffffffffu, k, o));
  return k;
}

// DEALT: a warp of its own for every chunk, the one of its number, in blocks of 64 threads; else as many warps as the chip holds, which
// take chunks from the counter.  The loop over chunks keeps so many values alive across a chunk that it spills 100 to 332 bytes at the 80
// registers of 24 warps per SM; without it nothing spills (2.45 M rows, 47 columns: 4.95 -> 3.36 ms, 3.53 in blocks of 256, 3.31 at 64
// registers with spills; 169 k, 40 columns 118 -> 94 us, 100, 97).  Chunks of narrow rows are too little work for a block's start
// (19.7 k rows, 3 columns: 20.8 by the counter, 23.2 dealt) unless the chip holds all of them at once.
template <int CL, bool DEALT>
__global__ void __launch_bounds__(DEALT ? 64 : 256, DEALT ? 12 : 3)
k_search_z_out(const int* __restrict__ col, const float* __restrict__ dinv, const float4* __restrict__ T, const float4* __restrict__ S,
               int ld4, float4* scratch, const SearchOut p) {
  constexpr int GROUPS = 32 / CL;
  const int lane = threadIdx.x & 31, grp = lane / CL, cl = lane & (CL - 1);
  do {
    int ch = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (!DEALT) {
      ch = 0;
      if (lane == 0) ch = atomicAdd(p.chunk_counter, 1);
      ch = __shfl_sync(0xffffffffu, ch, 0);
    }
    if (ch >= p.n_chunks) return;
    const SegChunk c = p.chunks[ch];
    if (__ldcg(&p.ctl[c.comm].done)) continue;   // skipped: none of its slots is filled
    double lin = 0.0, quad = 0.0;
    if (c.length > 0) {
      const SegRef* const segs = p.segs + c.first;
      if (c.length == 1) quad = short_segments<CL, 1, CL >= 8 ? 8 : CL>(segs, c.count, col, dinv, T, ld4, lane);
      else if (c.length == 2) quad = short_segments<CL, 2, CL >= 4 ? 4 : CL>(segs, c.count, col, dinv, T, ld4, lane);
      else if (c.length == 3) quad = short_segments<CL, 3, CL >= 2 ? 2 : CL>(segs, c.count, col, dinv, T, ld4, lane);
      else if (CL >= 8 && c.length < p.share_from) {
        if constexpr (CL >= 8) quad = group_segments<CL, 8>(segs, c.count, c.length, col, dinv, T, ld4, lane);
      } else if (c.length < p.share_from) {
        for (int k = grp; k < c.count; k += GROUPS) {
          const SegRef sg = segs[k];
          const float4 v = vscale(sg.dinv, walk_run<4>(sg.begin, sg.begin + c.length, 0, 1, col, dinv, T, ld4, cl));
          quad += (double)dot4(v, v);
        }
      } else {
        for (int k = 0; k < c.count; ++k) {
          const SegRef sg = segs[k];
          const float4 v = vscale(sg.dinv, add_sets<CL>(walk_run<4>(sg.begin, sg.begin + c.length, grp, GROUPS, col, dinv, T, ld4, cl)));
          if (grp == 0) quad += (double)dot4(v, v);
        }
      }
    } else if (c.length == 0) {
      const long long e1 = (long long)(c.first + c.count) * ld4;
#pragma unroll 2
      for (long long e = (long long)c.first * ld4 + lane; e < e1; e += 32) lin += (double)dot4(T[e], S[e]);
    } else {
      const int4 it = p.items[c.first], sp = p.split[c.count];   // a piece {row, first entry, one past the last} of a segment {.., first item, items}
      const float4 v = add_sets<CL>(walk_run<4>(it.y, it.z, grp, GROUPS, col, dinv, T, ld4, cl));
      if (grp == 0 && cl < ld4) scratch[(long long)c.first * ld4 + cl] = v;
      __threadfence();
      __syncwarp();
      int done = 0;
      if (lane == 0) done = atomicAdd(p.split_done + c.count, 1);
      done = __shfl_sync(0xffffffffu, done, 0);
      if (done + 1 < sp.w) continue;
      __threadfence();
      if (lane == 0) p.split_done[c.count] = 0;
      if (lane < ld4) {   // the pieces in item order
        float4 k;
        vzero(k);
        for (int q = 0; q < sp.w; ++q) k = vadd(k, __ldcg(scratch + (long long)(sp.z + q) * ld4 + lane));
        k = vscale(dinv[it.x], k);
        quad = (double)dot4(k, k);
      }
    }
    lin = warp_sum(lin);
    quad = warp_sum(quad);
    const int s0 = p.slot_ptr[c.comm], s1 = p.slot_ptr[c.comm + 1];
    int done = 0;
    if (lane == 0) {
      p.slots[2 * (size_t)c.slot] = lin;
      p.slots[2 * (size_t)c.slot + 1] = quad;
      __threadfence();
      done = atomicAdd(p.comm_done + c.comm, 1);
    }
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done + 1 < s1 - s0) continue;
    __threadfence();
    if (lane == 0) p.comm_done[c.comm] = 0;
    double sums[2] = {0.0, 0.0};
#pragma unroll 4
    for (int s = s0 + lane; s < s1; s += 32) {
      sums[0] += __ldcg(p.slots + 2 * (size_t)s);
      sums[1] += __ldcg(p.slots + 2 * (size_t)s + 1);
    }
    sums[0] = warp_sum(sums[0]);
    sums[1] = warp_sum(sums[1]);
    decide_one(p.ctl + c.comm, sums, p.own[c.comm * 3 + 2], p.a, p.n_active, p.status);
  } while (!DEALT);
}

// The move of the blocks after it: Z_l[i,:] <- Z_l[i,:] - G[i,:] / theta_{comm(i)} (Eq. 10), and the log entries.
__global__ void __launch_bounds__(256)
k_move_z(float4* __restrict__ Z, const float4* __restrict__ G, int ld4, long long n, const int* __restrict__ row_comm,
         const SearchCtl* __restrict__ ctl, int n_comm, const DecisionLog log, int* __restrict__ chunk_counter) {
  gtc::enter_kernel();
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  if (first == 0) *chunk_counter = 0;
  for (long long i = first; i < n_comm; i += stride) log_decision(log, (int)i, ctl + i);
  for (long long e = first; e < n * ld4; e += stride) {   // below 2^32
    const float s = ctl[row_comm[(unsigned)e / (unsigned)ld4]].inv_step;
    if (s == 0.f) continue;
    Z[e] = vfma(-s, G[e], Z[e]);
  }
}

// ------------------------------------------------------------------------------------------
// Output layer rows (Eq. 7) and the dual (Eq. 3).  q = row of A~ Z_{L-1}^k W_L^{k+1}.
//   training rows: FISTA on  loss_scale * CE(z, y) + <u, z - q> + (rho/2)||z - q||^2 ;  other rows: z = q - u / rho.
//   dual_now != 0: U <- u + rho (z_old - q) in the same sweep (Eq. 3 as printed).
// The first `train_blocks` blocks take the training rows (`rows` lists them), LPR lanes per row with CPL classes each (C <=
// LPR * CPL): a lane that holds several classes costs an exponential per class either way, but the two reductions per
// iteration then take log2(LPR) shuffles for 32 / LPR rows at once.  91 k rows x 40 classes x 30 iterations: a warp per row
// 255 us, 8 lanes per row 95 us.  The other blocks sweep the remaining rows elementwise.
// momentum[j] = (t_j - 1) / t_{j+1} of FISTA's sequence t_1 = 1, t_{j+1} = (1 + sqrt(1 + 4 t_j^2)) / 2: the same for every
// row, so it is tabulated once (in fp64).
// ------------------------------------------------------------------------------------------
struct OutputArgs {
  float *Z, *U;
  const float* H;
  int ld, C;
  long long n;
  const unsigned char* train;
  const int *rows, *y;
  int n_train, train_blocks;
  const float* momentum;
  float rho, loss_scale;
  int iters, dual_now, update_z;
};
template <int LPR, int CPL>
__global__ void __launch_bounds__(256)
k_output(const OutputArgs p) {
  gtc::enter_kernel();
  if ((int)blockIdx.x >= p.train_blocks) {
    const int ld4 = p.ld / 4;
    float4* const Z4 = reinterpret_cast<float4*>(p.Z);
    float4* const U4 = reinterpret_cast<float4*>(p.U);
    const float4* const H4 = reinterpret_cast<const float4*>(p.H);
    const float inv_rho = 1.f / p.rho;
    const long long total = p.n * ld4;   // below 2^32
    for (long long e = (long long)(blockIdx.x - p.train_blocks) * blockDim.x + threadIdx.x; e < total;
         e += (long long)(gridDim.x - p.train_blocks) * blockDim.x) {
      if (p.train[(unsigned)e / (unsigned)ld4]) continue;
      const float4 q = H4[e], u = U4[e];
      if (p.dual_now) {
        const float4 z = Z4[e];
        U4[e] = make_float4(fmaf(p.rho, z.x - q.x, u.x), fmaf(p.rho, z.y - q.y, u.y), fmaf(p.rho, z.z - q.z, u.z),
                            fmaf(p.rho, z.w - q.w, u.w));
      }
      if (p.update_z)
        Z4[e] = make_float4(fmaf(-u.x, inv_rho, q.x), fmaf(-u.y, inv_rho, q.y), fmaf(-u.z, inv_rho, q.z), fmaf(-u.w, inv_rho, q.w));
    }
    return;
  }
  constexpr int kTable = 128;          // iterations whose momentum is kept in shared memory
  __shared__ float s_mom[kTable];
  for (int k = threadIdx.x; k < min(p.iters, kTable); k += blockDim.x) s_mom[k] = p.momentum[k];
  __syncthreads();
  const int lane = threadIdx.x & (LPR - 1);
  const int slot = (int)((blockIdx.x * blockDim.x + threadIdx.x) / LPR);
  const bool here = slot < p.n_train;   // lanes without a row keep step with the shuffles of the others
  const int row = here ? p.rows[slot] : 0;
  const int C = here ? p.C : 0;
  float q[CPL], u[CPL], z[CPL];
  const long long base = (long long)row * p.ld;
#pragma unroll
  for (int t = 0; t < CPL; ++t) {
    const int c = lane + LPR * t;
    q[t] = u[t] = z[t] = 0.f;
    if (c < C) { q[t] = p.H[base + c]; u[t] = p.U[base + c]; z[t] = p.Z[base + c]; }
  }
  if (p.dual_now) {
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const int c = lane + LPR * t;
      if (c < C) p.U[base + c] = fmaf(p.rho, z[t] - q[t], u[t]);
    }
  }
  if (!p.update_z) return;
  const int yi = here ? p.y[row] : -1;
  const float step = 1.f / (0.5f * p.loss_scale + p.rho);
  float xp[CPL], v[CPL];
#pragma unroll
  for (int t = 0; t < CPL; ++t) { xp[t] = z[t]; v[t] = z[t]; }
  for (int it = 0; it < p.iters; ++it) {
    float mx = -3.0e38f;
#pragma unroll
    for (int t = 0; t < CPL; ++t)
      if (lane + LPR * t < C) mx = fmaxf(mx, v[t]);
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float ex[CPL], se = 0.f;
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      ex[t] = (lane + LPR * t < C) ? expf(v[t] - mx) : 0.f;
      se += ex[t];
    }
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    const float inv_se = 1.f / se;
    const float mom = it < kTable ? s_mom[it] : p.momentum[it];
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const float pr = ex[t] * inv_se - (lane + LPR * t == yi ? 1.f : 0.f);
      const float g = p.loss_scale * pr + u[t] + p.rho * (v[t] - q[t]);
      const float x = fmaf(-step, g, v[t]);
      v[t] = fmaf(mom, x - xp[t], x);
      xp[t] = x;
    }
  }
#pragma unroll
  for (int t = 0; t < CPL; ++t) {
    const int c = lane + LPR * t;
    if (c < C) p.Z[base + c] = xp[t];
  }
}

// ------------------------------------------------------------------------------------------
// Reporting (Eq. 1) and the forward pass of Problem 1.
// ------------------------------------------------------------------------------------------
// Every sum is formed in one launch: a block leaves its N totals in partial[b * N ..], and the last block to finish (ticket, left at
// zero) adds the blocks' up thread-strided and by the block tree, whichever block that is: the same bits from run to run.  out[j] = the
// sum, or += where `more`.
template <int N>
__device__ __forceinline__ void add_up(double (&v)[N], double* sh, double* partial, unsigned* ticket, double* __restrict__ out, bool more) {
  __shared__ int s_last;
  block_sums(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) partial[(size_t)blockIdx.x * N + j] = v[j];
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = 0.0;
#pragma unroll 4
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] += __ldcg(partial + (size_t)b * N + j);
  block_sums(v, sh);
  if (threadIdx.x == 0) {
    *ticket = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) out[j] = more ? out[j] + v[j] : v[j];
  }
}

// sum (z - f(h))^2
__global__ void __launch_bounds__(256)
k_sum_hidden_penalty(const float4* __restrict__ Z, const float4* __restrict__ H, long long n4, double* partial, unsigned* ticket,
                     double* __restrict__ out, bool more) {
  gtc::enter_kernel();
  __shared__ double sh[8];
  double s[1] = {0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (long long)gridDim.x * blockDim.x) {
    const float4 z = Z[i], h = H[i];
    const float a = z.x - relu(h.x), b = z.y - relu(h.y), c = z.z - relu(h.z), d = z.w - relu(h.w);
    s[0] += (double)(a * a + b * b + c * c + d * d);
  }
  add_up(s, sh, partial, ticket, out, more);
}

// <U, Z - H> and ||Z - H||^2
__global__ void __launch_bounds__(256)
k_sum_constraint(const float4* __restrict__ Z, const float4* __restrict__ H, const float4* __restrict__ U, long long n4, double* partial,
                 unsigned* ticket, double* __restrict__ out) {
  gtc::enter_kernel();
  __shared__ double sh[16];
  double s[2] = {0.0, 0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (long long)gridDim.x * blockDim.x) {
    const float4 z = Z[i], h = H[i], u = U[i];
    const float a = z.x - h.x, b = z.y - h.y, c = z.z - h.z, d = z.w - h.w;
    s[0] += (double)(u.x * a + u.y * b + u.z * c + u.w * d);
    s[1] += (double)(a * a + b * b + c * c + d * d);
  }
  add_up(s, sh, partial, ticket, out, false);
}

// Per row: cross-entropy of the row of Zrows with its label (training rows only); argmax of the row of `logits` (lowest index on
// ties) to labels[perm[row]], the caller's order; whether a training row's argmax equals its label.  out[0] = the cross-entropy sum,
// out[1] = the hits; out may be NULL, and so may either of Zrows / logits.  Eight lanes share a row (a warp per row and a partial sum
// for every eight rows, which one block then added up, took 44 + 21 us at 169 k rows of 40 classes; this 11).
__global__ void __launch_bounds__(256)
k_row_loss_argmax(const float4* __restrict__ Zrows, const float4* __restrict__ logits, int ld4, int C, int n,
                  const int* __restrict__ y, const unsigned char* __restrict__ train, int* __restrict__ labels,
                  const int* __restrict__ perm, double* partial, unsigned* ticket, double* __restrict__ out) {
  gtc::enter_kernel();
  __shared__ double sh[16];
  const int sub = threadIdx.x & 7;
  const unsigned lanes = 0xffu << (threadIdx.x & 24);
  double s[2] = {0.0, 0.0};
  for (int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3); row < n; row += (int)((gridDim.x * blockDim.x) >> 3)) {
    const long long base = (long long)row * ld4;
    const bool tr = train[row] != 0;
    if (Zrows != nullptr && tr) {
      float mx = -3.0e38f, at_label = 0.f, se = 0.f;
      const int label = y[row];
      for (int f = sub; f < ld4; f += 8) {
        const float4 v = Zrows[base + f];
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * f + k < C) {
            mx = fmaxf(mx, x[k]);
            if (4 * f + k == label) at_label = x[k];
          }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(lanes, mx, o));
        at_label += __shfl_xor_sync(lanes, at_label, o);   // one lane holds it, the others zero
      }
      for (int f = sub; f < ld4; f += 8) {
        const float4 v = Zrows[base + f];
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * f + k < C) se += expf(x[k] - mx);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) se += __shfl_xor_sync(lanes, se, o);
      if (sub == 0) s[0] += (double)(mx + logf(se) - at_label);
    }
    if (logits != nullptr) {
      float best = -3.0e38f;
      int arg = 0x7fffffff;
      for (int f = sub; f < ld4; f += 8) {
        const float4 v = logits[base + f];
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * f + k < C && x[k] > best) { best = x[k]; arg = 4 * f + k; }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(lanes, best, o);
        const int oa = __shfl_xor_sync(lanes, arg, o);
        if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
      }
      if (sub == 0 && labels) labels[perm[row]] = arg;
      if (sub == 0 && tr && arg == y[row]) s[1] += 1.0;
    }
  }
  if (out != nullptr) add_up(s, sh, partial, ticket, out, false);
}

// Y = relu(X) for n rows of ld4 float4, a warp per row.  row_max (may be NULL): the largest element of every row of Y.
__global__ void __launch_bounds__(256)
k_relu(const float4* __restrict__ X, float4* __restrict__ Y, int ld4, long long n, float* __restrict__ row_max) {
  const int lane = threadIdx.x & 31;
  for (long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += ((long long)gridDim.x * blockDim.x) >> 5) {
    float m = 0.f;
#pragma unroll 2
    for (int f = lane; f < ld4; f += 32) {
      const float4 y = vrelu(X[row * ld4 + f]);
      Y[row * ld4 + f] = y;
      m = fmaxf(m, vabsmax(y));
    }
    if (row_max == nullptr) continue;
    m = warp_max(m);
    if (lane == 0) row_max[row] = m;
  }
}

// out[row] = the largest magnitude of the row, a warp per row of ld4 float4.
__global__ void __launch_bounds__(256)
k_row_max(const float4* __restrict__ X, int ld4, long long n, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += ((long long)gridDim.x * blockDim.x) >> 5) {
    float m = 0.f;
#pragma unroll 4
    for (int f = lane; f < ld4; f += 32) m = fmaxf(m, vabsmax(X[row * ld4 + f]));
    m = warp_max(m);
    if (lane == 0) out[row] = m;
  }
}

// U <- U + rho (Z - H)
__global__ void k_dual(float4* __restrict__ U, const float4* __restrict__ Z, const float4* __restrict__ H,
                       long long n4, float rho) {
  gtc::enter_kernel();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (long long)gridDim.x * blockDim.x) {
    float4 u = U[i];
    const float4 z = Z[i], h = H[i];
    u.x = fmaf(rho, z.x - h.x, u.x); u.y = fmaf(rho, z.y - h.y, u.y);
    u.z = fmaf(rho, z.z - h.z, u.z); u.w = fmaf(rho, z.w - h.w, u.w);
    U[i] = u;
  }
}

// The tables of k_spmm_sets' rows and of the caller's columns (may be NULL) from those of the graph.
__global__ void k_gather_tables(const int* __restrict__ order, const int* __restrict__ row_ptr, const float* __restrict__ dinv, int n,
                                int4* __restrict__ row_table, const int* __restrict__ col, const int* __restrict__ perm, long long nnz,
                                int* __restrict__ user_col) {
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < n; i += stride) {
    const int row = order[i];
    row_table[i] = make_int4(row, row_ptr[row], row_ptr[row + 1], __float_as_int(dinv[row]));
  }
  if (user_col == nullptr) return;
  for (long long e = first; e < nnz; e += stride) user_col[e] = perm[col[e]];
}

// dst[c][r] = src[r][c] for a small rows x cols matrix (weights and their gradients).
__global__ void k_transpose_small(const float* __restrict__ src, int lds, float* __restrict__ dst, int ldd, int rows,
                                  int cols) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * cols) return;
  const int r = e / cols, c = e % cols;
  dst[c * ldd + r] = src[r * lds + c];
}

// What the images of a weight matrix are scaled and marked by: {largest finite magnitude, smallest above zero, both as bits, whether there is
// a zero}.  An infinity or NaN stays in its column of the product under any scale and counts for nothing.
struct WeightRange {
  unsigned most, least;
  int zero, pad;
};
// All threads of a block of 256: the range of what they hold.
__device__ __forceinline__ WeightRange block_range(WeightRange w) {
  __shared__ WeightRange s_range[8];
  w.most = __reduce_max_sync(0xffffffffu, w.most);
  w.least = __reduce_min_sync(0xffffffffu, w.least);
  w.zero = __any_sync(0xffffffffu, w.zero);
  if ((threadIdx.x & 31) == 0) s_range[threadIdx.x >> 5] = w;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    w.most = max(w.most, s_range[k].most);
    w.least = min(w.least, s_range[k].least);
    w.zero |= s_range[k].zero;
  }
  return w;
}
constexpr unsigned kLargestBits = 0x7f7fffffu;   // of FLT_MAX
// One range per block of at most 256, added up by k_load_weight (on the host, before: 64,000 elements 51 to 118 us).
__global__ void __launch_bounds__(256)
k_weight_range(const float* __restrict__ src, long long count, WeightRange* __restrict__ out) {
  WeightRange w{0u, kLargestBits, 0, 0};
#pragma unroll 4
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const unsigned size = __float_as_uint(src[i]) & 0x7fffffffu;
    w.most = max(w.most, size <= kLargestBits ? size : 0u);
    w.least = min(w.least, size > 0u ? size : kLargestBits);
    w.zero |= size == 0u;
  }
  w = block_range(w);
  if (threadIdx.x == 0) out[blockIdx.x] = w;
}

// W (rows x cols, leading dimension ldw), its transpose and its images from a dense matrix; padding columns become zero.  ranges:
// what k_weight_range left of it, where an image is kept.
__global__ void __launch_bounds__(256)
k_load_weight(const float* __restrict__ src, int rows, int cols, float* __restrict__ W, int ldw,
              float* __restrict__ Wt, int ldwt, const gtc::Image image, const gtc::Image image_t, const WeightRange* __restrict__ ranges, int n_ranges) {
  const WeightRange own = (int)threadIdx.x < n_ranges ? ranges[threadIdx.x] : WeightRange{0u, kLargestBits, 0, 0}, range = block_range(own);
  const float bound = __uint_as_float(range.most), least = __uint_as_float(range.least), scale = gtc::scale_of(bound);
  if (blockIdx.x == 0) {
    // the bound is scaled to 2^14 at least: elements below 2^-27 of it may be too small for a pair, below 2^-22 they make the matrix wide
    const int marks = ((double)least < (double)bound * 0x1p-27 || least < FLT_MIN ? gtc::kBelowPairs : 0) |
                      (range.zero || (double)least < (double)bound * 0x1p-22 ? gtc::kWide : 0);
    gtc::put_scales(image, cols, bound);
    gtc::put_scales(image_t, rows, bound);
    gtc::put_marks(image, cols, marks);
    gtc::put_marks(image_t, rows, marks);
  }
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < (long long)rows * ldw; i += stride) {
    const long long r = i / ldw, c = i - r * ldw;
    const float w = c < cols ? src[r * cols + c] : 0.f;
    W[i] = w;
    if (c < cols) {
      gtc::put_half(image, (int)c, (int)r, w * scale);
      gtc::put_half(image_t, (int)r, (int)c, w * scale);
    }
  }
  for (long long i = first; i < (long long)cols * ldwt; i += stride) {
    const long long c = i / ldwt, r = i - c * ldwt;
    Wt[i] = r < rows ? src[r * cols + c] : 0.f;
  }
}

__global__ void k_put_steps(SearchCtl* __restrict__ ctl, const double* __restrict__ values, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) ctl[i].t_prev = values[i];
}
__global__ void k_take_steps(const SearchCtl* __restrict__ ctl, double* __restrict__ values, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) values[i] = ctl[i].t_prev;
}

// dst[r] = src[rows[r]] for padded rows of ld4 float4: the staging copy of the rows a rank does not own
// (what a receive from their owners would deliver) behind its own rows.
__global__ void k_gather_rows(const float4* __restrict__ src, const int* __restrict__ rows, float4* __restrict__ dst,
                              int ld4, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count * ld4;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / ld4;
    dst[i] = src[(long long)rows[r] * ld4 + (i - r * ld4)];
  }
}

// Row gather / scatter between the caller's dense layout (original order, width C) and the internal one (community order,
// leading dimension ld, padding columns zero).  `inv`: original id -> new id.  Both directions walk the caller's matrix in
// its order, so that it can lie in host memory (reads and writes over the bus are then whole lines); the scattered side is
// the device's own.
template <typename I>
__device__ __forceinline__ void permute_rows(const float* __restrict__ src, float* __restrict__ dst, const int* __restrict__ inv,
                                             I n, I C, I ld, int to_internal) {
  const I first = (I)blockIdx.x * blockDim.x + threadIdx.x, stride = (I)gridDim.x * blockDim.x;
  if (to_internal) {
    for (I e = first; e < n * ld; e += stride) {
      const I r = e / ld, c = e - r * ld;
      dst[(long long)inv[r] * ld + c] = c < C ? src[(long long)r * C + c] : 0.f;
    }
  } else {
    for (I e = first; e < n * C; e += stride) {
      const I r = e / C, c = e - r * C;
      dst[e] = src[(long long)inv[r] * ld + c];
    }
  }
}
__global__ void k_permute_rows(const float* __restrict__ src, float* __restrict__ dst, const int* __restrict__ inv,
                               long long n, int C, int ld, int to_internal) {
  if (n * ld + (long long)gridDim.x * blockDim.x < (1LL << 32))   // 32-bit divisions
    permute_rows<unsigned>(src, dst, inv, (unsigned)n, (unsigned)C, (unsigned)ld, to_internal);
  else permute_rows<long long>(src, dst, inv, n, C, ld, to_internal);
}

}  // namespace gk
