// C-ABI library of the community-based ADMM GCN trainer: host orchestration of the kernels in
// kernels.cuh.  See include/gcn_admm.h for the contract of every entry point.
#include "../../include/gcn_admm.h"

#include <climits>
#include <cmath>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "gemm_half.cuh"
#include "gemm_tc.cuh"
#include "graph_index.hpp"
#include "kernels.cuh"
#include "memory.hpp"
#include "shard_plan.hpp"

using gcn_admm_host::GraphIndex;

namespace {
// Named range on the profiler timeline (NVTX; a no-op unless a tool is attached) for the life of the object.
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
};
}  // namespace
using gk::SearchCtl;

namespace {

constexpr int kLogPasses = 256;
constexpr int kSmCount = 148;
constexpr long long kHalfMinRows = 16384;    // row count from which products of any width go by split halves
constexpr int kZBlockRows = 32;      // rows per block of the hidden-layer gradient's closing sweep
constexpr int kChunkGroups = 512;    // groups the sums of a scoring sweep's chunks are first added up in, when there are more chunks
constexpr long long kUserColumns = 16 << 20;  // entries up to which a handle keeps the caller's column numbers too (64 MB)
constexpr size_t kDirectBytes = (size_t)256 << 10;   // matrices up to this size cross the bus inside the permuting kernel (one copy and its latency less)
constexpr long long kSmallProblem = 1LL << 27;   // nodes x widest layer: below it launch gaps show in a pass
// Stored entries one warp walks before a row is cut into items, where the caller leaves it open.  A warp that walks a long row alone
// outlasts a launch whose warps have few entries each, and every cut costs an item's sums written, read and added up; the line
// lies where the two meet, the lower the fewer entries a resident warp has, and well above the mean row (at twice it few rows are
// cut).  us at 32 / 48 / 64 / 96 / 128 / 256 entries: 13 k rows, 0.15 M entries, six passes 2761 / 2757 / 2761 / 2806 / 2867 / 3099;
// 23 k, 0.12 M, objective curve 769 / 782 / 788 / 815 / 833 / 935; 30 k, 0.51 M, serial 2270 / 2244 / 2247 / 2255 / 2289 / 2454;
// 47 k, 1.6 M 3891 / 3762 / 3691 / 3688 / 3730 / 3921; 169 k, 2.5 M 10983 / 10834 / 10689 / 10689 / 10826 / 10868; 239 k, 6.7 M
// 2631 / 2474 / 2380 / 2327 / 2325 / 2330; 409 k, 12.4 M 3720 / 3358 / 3185 / 3019 / 2956 / 2867.  127 k rows of 46 entries lose at 64.
// Under 4,096 rows a launch is a wave of short chains and no length differs from 256 by more than its runs do.
int default_long_row(long long n, long long nnz) {
  if (n < 4096 || nnz > 8000000) return 256;
  const int line = nnz <= 300000 ? 48 : nnz <= 2000000 ? 64 : 96;
  return (int)std::min<long long>(256, std::max<long long>(line, 2 * nnz / n));
}

thread_local std::string g_create_error;

inline int ldpad(int c) { return (c + 3) & ~3; }
constexpr int kMaxWidth = 1 << 24;   // widest matrix an entry point accepts (keeps the padded width inside int)

// Output function of the splitmix64 generator applied to the state x + 0x9E3779B97F4A7C15.
inline unsigned long long splitmix64(unsigned long long x) {
  unsigned long long z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
inline long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

struct Fail {
  int code;
  std::string msg;
};

#define CU(expr)                                                                           \
  do {                                                                                     \
    cudaError_t e__ = (expr);                                                              \
    if (e__ != cudaSuccess)                                                                \
      throw Fail{GCN_ADMM_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e__)};  \
  } while (0)

template <typename T>
T* dalloc(size_t count) {
  void* p = nullptr;
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e == cudaSuccess) e = gcn_admm_mem::Pool::get().allocate(device, std::max<size_t>(count, 1) * sizeof(T), &p);
  if (e != cudaSuccess)
    throw Fail{e == cudaErrorMemoryAllocation ? GCN_ADMM_ERR_ALLOC : GCN_ADMM_ERR_CUDA,
               std::string("cudaMalloc: ") + cudaGetErrorString(e)};
  return static_cast<T*>(p);
}

// cuTensorMapEncodeTiled, looked up through the runtime (the library does not link the driver API directly).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// Tensor map of a row-major rows x ld fp32 matrix for 128-row x 32-column tiles written with the 128-byte
// swizzle; elements outside the matrix read as zero.  False when the map cannot be made (the product then takes the
// form that stages the operand through registers).
bool make_a_tile_map(const float* A, long long rows, int ld, CUtensorMap* map) {
  EncodeTiledFn fn = encode_tiled();
  if (fn == nullptr) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)gtc::kChunkK, (cuuint32_t)gtc::kBlockM};
  const cuuint32_t elem[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(A), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Lets `kernel` be launched on the current device (`device`) with `smem` bytes of dynamic shared memory.  The limit belongs to the
// function, not to a handle, and handles of other sizes are stepped in between: it is only ever raised.  (What needs no leave is 48
// KB, the kernel's static shared memory among them.)
void allow_shared(int device, const void* kernel, size_t smem) {
  static std::mutex mutex;
  static std::map<std::pair<int, const void*>, size_t> most;
  std::lock_guard<std::mutex> lock(mutex);
  size_t& limit = most[{device, kernel}];
  limit = std::max(limit, smem);
  if (limit > 40 * 1024) CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
}

bool is_device_pointer(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

struct ProfStat {
  long long launches = 0;
  double ms = 0.0, bytes = 0.0, flops = 0.0;
};
struct ProfPending {
  ProfStat* stat;
  cudaEvent_t a, b;
};

struct gcn_admm {
  gcn_admm_params p{};
  // launch accounting: every kernel launch goes through a Scope (below)
  long long launches = 0;
  bool profiling = false;
  std::map<std::string, ProfStat> prof;
  std::vector<ProfPending> pending;
  std::vector<cudaEvent_t> event_pool;
  cudaEvent_t get_event() {
    if (!event_pool.empty()) { cudaEvent_t e = event_pool.back(); event_pool.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
  }
  // Counts `kernels` launches; when profiling, brackets them with events on the handle's stream and
  // books the algorithmic bytes / flops of the work under `name`.
  struct Scope {
    gcn_admm* h;
    cudaEvent_t b = nullptr;
    Scope(gcn_admm* h_, const char* name, int kernels, double bytes, double flops) : h(h_) {
      h->launches += kernels;
      if (!h->profiling) return;
      ProfStat& st = h->prof[name];
      st.launches += kernels;
      st.bytes += bytes;
      st.flops += flops;
      cudaEvent_t a = h->get_event();
      b = h->get_event();
      cudaEventRecord(a, h->stream);
      h->pending.push_back(ProfPending{&st, a, b});
    }
    ~Scope() { if (b) cudaEventRecord(b, h->stream); }
  };
  void collect_profile() {
    cudaStreamSynchronize(stream);
    event_pool.reserve(event_pool.size() + 2 * pending.size());
    for (ProfPending& q : pending) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, q.a, q.b) == cudaSuccess) q.stat->ms += ms;
      event_pool.push_back(q.a);
      event_pool.push_back(q.b);
    }
    pending.clear();
  }

  cudaStream_t stream = nullptr;
  int L = 0;
  long long n = 0;
  int M = 0;
  int n_train = 0;
  std::vector<int> C, ld;   // widths C_0..C_L and their padded leading dimensions
  int max_ld = 0;
  GraphIndex gi;
  gcn_admm_mem::Slab slab;                 // device memory: everything but wide_sums
  gcn_admm_mem::Stage stage;               // page-locked staging of host buffers

  int *d_row_ptr = nullptr, *d_col = nullptr, *d_row_comm = nullptr, *d_perm = nullptr, *d_inv = nullptr;
  int* d_y = nullptr;
  float* d_dinv = nullptr;
  unsigned short* d_col_comm = nullptr;   // community of every stored column
  // rows too long for one warp, cut into items (see gcn_admm_host::LongRowTables)
  int4 *d_items = nullptr, *d_split = nullptr, *d_long_rows = nullptr;
  int *d_item_row = nullptr, *d_row_done = nullptr;   // long row of every item; per long row a counter of finished items
  int n_items = 0, n_split = 0, n_long = 0, long_len = 0;
  float* item_sums = nullptr;             // n_items x max_ld
  size_t item_sums_elems = 0;
  gcn_admm_mem::Slab wide_sums;           // the same for the widest matrix gcn_admm_propagate was given, where that is wider than every layer
  unsigned char* d_train = nullptr;
  int* d_train_rows = nullptr;            // new ids of the training rows, ascending
  float* d_fista_momentum = nullptr;      // (t_j - 1) / t_{j+1}, j = 1..fista_iters

  std::vector<float*> W, Wt, Z, P, H;   // 1..L
  float* U = nullptr;
  float *B0 = nullptr, *B1 = nullptr, *B2 = nullptr;   // N x max_ld scratch
  float* grad = nullptr;     // max over l of C_{l-1} x ld_l
  float* grad_t = nullptr;   // its transpose, C_l x ld_{l-1} (K-major operand of the tensor-core product)
  int* tc_error = nullptr;   // &report->error: raised by a tensor-core product (1) or a search (2) whose bounded wait ran out
  std::vector<gtc::Image> img_H, img_G, img_D;   // 1..L: images of W_l for P_l W_l, of W_l for S W_l^T, of the gradient for P_l grad
  std::vector<float*> P_max;                     // 1..L: row maxima of P_l; NULL where no product of it takes them
  float *B1_max = nullptr, *B2_max = nullptr;    // of S and G (B1, B2) while a Z update uses them, of the forward pass's operands
  float* part = nullptr;     // split partial sums of the transposed product
  size_t part_elems = 0;
  SearchCtl *ctl_w = nullptr, *ctl_z = nullptr;   // [L+1], [(L+1) * M]
  double* sums_z = nullptr;
  gk::Report* report = nullptr;             // objective sums and error flags
  double* red_part = nullptr;               // per-block partial sums awaiting their fixed-order reduction
  int4* d_zblocks = nullptr;                // row blocks of at most kZBlockRows rows, none crossing a community, and that community
  unsigned *ticket = nullptr, *tile_tickets = nullptr, *comm_tickets = nullptr;   // counters of finished blocks (one launch; per community), zero between launches
  gk::GridBar* grid_bar = nullptr;          // meeting point of the cooperative launches (one at a time: one stream)
  int* d_comm_block_ptr = nullptr;          // [M+1] first row block of every community
  int n_zblocks = 0;
  int *d_h1_age = nullptr, *skip_h1 = nullptr;   // see k_end_pass
  float *RL = nullptr, *DL = nullptr;       // the last layer's R and P grad, where its chain runs beside the hidden layers' (see Lane)
  int *n_active = nullptr, *status = nullptr, *d_pass = nullptr;   // status = &report->status
  // Z scoring: units in chunks of about equally many stored entries, dealt to the warps of the grid in a fixed order
  int* d_chunk_ptr = nullptr;
  int* d_row_order = nullptr;               // rows per community by falling length, for d_row_table at create
  int4* d_row_table = nullptr;              // the same order with what those kernels want of a row (see k_spmm_sets)
  int* d_user_col = nullptr;                // the caller's row of every column; NULL on graphs of more than kUserColumns entries
  // closed-form search of the last hidden layer (gcn_admm_host::SegmentTables)
  gk::SegRef* d_segs = nullptr;
  gk::SegChunk* d_seg_chunks = nullptr;
  int *d_slot_ptr = nullptr, *comm_done = nullptr, *split_done = nullptr;
  double* slots = nullptr;
  int n_seg_chunks = 0;
  int n_chunks = 0;
  double* z_chunk_part = nullptr;           // [chunk][M][candidates] sums of one sweep, per chunk of units
  double* z_group_part = nullptr;           // [group of chunks][M][candidates], chunks added in order
  int* chunk_counter = nullptr;             // hands the chunks out to the warps of a sweep
  double* split_scores = nullptr;           // [n_split][candidates] sums of the segments scored in pieces
  int *d_split_order = nullptr, *d_split_ptr = nullptr;   // split entries grouped by community
  cudaGraphExec_t pass_graph = nullptr;   // one pass of Algorithm 1, recorded once and replayed
  long long single_passes = 0;            // passes launched without it
  int *log_trial_w = nullptr, *log_trial_z = nullptr;
  double *log_q_w = nullptr, *log_q_z = nullptr;
  long long log_count = 0;
  long long launches_per_pass = 0;
  bool fresh = false;        // P_l, H_l agree with the stored W, Z
  std::string err;
  std::vector<int> ix_cache[16];
  gcn_admm_host::ShardPlan shard_plan;      // last plan asked for (host only)
  std::vector<int> shard_ranges;

  // Device memory is asked for first and cut from one slab by commit(): tables to upload (staged in one stream of copies),
  // then what starts at zero, then the rest.  The sources must live until commit() returns.
  enum Start { kTable, kZero, kPlain };
  struct Want {
    void** slot;
    size_t bytes;
    const void* src;
    Start start;
  };
  std::vector<Want> wants;
  // Counters that every complete launch leaves at zero for the next one, and their sizes: zeroed by check() after one that gave up.
  std::vector<std::pair<void**, size_t>> counters;
  template <typename T>
  void want_counter(T*& slot, size_t count) {
    want(slot, count, kZero);
    counters.push_back({reinterpret_cast<void**>(&slot), std::max<size_t>(count, 1) * sizeof(T)});
  }
  template <typename T>
  void want(T*& slot, size_t count, Start start = kPlain) {
    wants.push_back(Want{reinterpret_cast<void**>(&slot), std::max<size_t>(count, 1) * sizeof(T), nullptr, start});
  }
  template <typename T, typename V>
  void want_table(T*& slot, const V& v) {
    static_assert(sizeof(T) == sizeof(typename V::value_type), "a table is uploaded as it is");
    wants.push_back(Want{reinterpret_cast<void**>(&slot), std::max<size_t>(v.size(), 1) * sizeof(T), v.empty() ? nullptr : v.data(), kTable});
  }
  gcn_admm_mem::Slab take_slab(size_t bytes) {
    gcn_admm_mem::Slab slab;
    const cudaError_t e = gcn_admm_mem::Pool::get().take(p.device, bytes, &slab);
    if (e != cudaSuccess)
      throw Fail{e == cudaErrorMemoryAllocation ? GCN_ADMM_ERR_ALLOC : GCN_ADMM_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e)};
    return slab;
  }
  void commit() {
    std::stable_sort(wants.begin(), wants.end(), [](const Want& a, const Want& b) { return a.start < b.start; });
    size_t total = 0, zero_begin = 0, zero_end = 0;
    std::vector<size_t> at;
    for (const Want& w : wants) {
      if (w.start == kZero && zero_end == 0) zero_begin = total;
      at.push_back(total);
      total += (w.bytes + 255) / 256 * 256;
      if (w.start == kZero) zero_end = total;
    }
    slab = take_slab(total);
    char* const base = slab.base;
    for (size_t k = 0; k < wants.size(); ++k) {
      *wants[k].slot = base + at[k];
      if (wants[k].start == kTable && wants[k].src) CU(stage.put(base + at[k], wants[k].src, wants[k].bytes, stream));
    }
    CU(stage.flush(stream));
    if (zero_end > zero_begin) CU(cudaMemsetAsync(base + zero_begin, 0, zero_end - zero_begin, stream));
    wants.clear();
  }
  int grid_for(long long work_items, int per_block = 256) const {
    return (int)std::max<long long>(1, std::min<long long>(cdiv(work_items, per_block), (long long)kSmCount * 8));
  }

  // ---- launches -----------------------------------------------------------------------
  // out_max: where the row maxima of the result go, or NULL
  void spmm(const float* x, float* out, int ldx, float* out_max, bool relu = false) {
    char name[48];
    std::snprintf(name, sizeof name, "spmm@%d", ldx);
    Scope sc(this, name, 1, 4.0 * gi.nnz + 8.0 * n + 8.0 * (double)n * ldx, 2.0 * (double)gi.nnz * ldx);
    if (relu) spmm_tables<4, false, true>(gather_graph(ldx), x, out, ldx / 4, out_max);
    else spmm_tables<4, false>(gather_graph(ldx), x, out, ldx / 4, out_max);
    if (out_max != nullptr && ldx > 256) {   // its rows are shared by blocks
      launch_alone(gk::k_row_max, grid_for(32 * n), 256, 0, (const float4*)out, ldx / 4, n, out_max);
      CU(cudaGetLastError());
      ++launches;
    }
  }

  // out = A~ x for dense n x width device matrices in the caller's row order, in vectors as wide as the width and
  // both addresses allow.  `wide`: long rows may go through wide_sums; the caller then waits for the result.
  void propagate_dense(const float* x, int width, float* out, bool wide) {
    char name[48];
    std::snprintf(name, sizeof name, "spmm@%d", ldpad(width));
    Scope sc(this, name, 1, 4.0 * gi.nnz + 8.0 * n + 8.0 * (double)n * width, 2.0 * (double)gi.nnz * width);
    const GatherGraph g = gather_graph(ldpad(width), wide);
    const uintptr_t low = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(out) | ((uintptr_t)width * sizeof(float));
    if ((low & 15) == 0) spmm_tables<4, true>(g, x, out, width / 4);
    else if ((low & 7) == 0) spmm_tables<2, true>(g, x, out, width / 2);
    else spmm_tables<1, true>(g, x, out, width);
  }

  // The handle's graph for a propagation of ldw padded columns.  Long rows go as items unless the operand is
  // wider than the item buffer (a caller's matrix wider than every layer, where nothing may be allocated): then
  // they are walked whole, slower but the same sums.
  struct GatherGraph {
    const int *row_ptr, *col, *perm, *user_col;
    const float* dinv;
    const int4 *row_table, *items, *rows;
    const int* item_row;
    int* row_done;
    int n, n_items, n_long, long_len;
    float* item_sums;
  };
  GatherGraph gather_graph(int ldw, bool wide = false) const {
    const size_t need = (size_t)n_items * ldw;
    float* const room = need <= item_sums_elems ? item_sums : wide && need * sizeof(float) <= wide_sums.size ? reinterpret_cast<float*>(wide_sums.base) : nullptr;
    const bool cut = n_items > 0 && room != nullptr;
    return GatherGraph{d_row_ptr, d_col, d_perm, d_user_col, d_dinv, d_row_table, d_items, d_long_rows, d_item_row, d_row_done,
                       (int)n, cut ? n_items : 0, cut ? n_long : 0, cut ? long_len : INT_MAX, room};
  }
  // Room for the items' sums at ldw padded columns.  Passes, recorded ones too, and callers under capture hold item_sums, which
  // therefore stays what it is; wide_sums serves calls that wait for their result, so a larger one may take its place.
  void grow_wide_sums(int ldw) {
    const size_t need = (size_t)n_items * ldw;
    if (need <= item_sums_elems || need * sizeof(float) <= wide_sums.size) return;
    CU(cudaStreamSynchronize(stream));
    gcn_admm_mem::Pool::get().give(wide_sums);
    wide_sums = gcn_admm_mem::Slab{};
    wide_sums = take_slab(need * sizeof(float));
  }

  template <typename T> struct Same { using type = T; };   // keeps a parameter out of template deduction
  // Launch of a kernel that waits for its predecessor on the stream itself (gtc::enter_kernel), where the grid is short, so
  // that the launch is a good part of its time.  In a pass that is a wave or less: waiting blocks hold their SMs' threads
  // against what still runs there and against the other line of launches (without the bound 13.8 k rows lost 3 %, 169 k
  // 1 %).  A propagation on its own has nothing beside it (2.7 k rows, 16 columns, call after call: 6.1 -> 4.0 us).  The first
  // kernel after a wait for the other line's event takes the ordinary dependency on both.
  template <typename... Args>
  void launch(void (*kernel)(Args...), dim3 grid, int threads, size_t smem, typename Same<Args>::type... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute behind{};
    behind.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    behind.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &behind;
    cfg.numAttrs = joined || (long long)grid.x * grid.y * grid.z > (in_pass ? 4 : 32) * kSmCount ? 0 : 1;
    joined = false;
    CU(cudaLaunchKernelEx(&cfg, kernel, args...));
  }
  // The ordinary launch, for kernels without that wait: the products (with it 13.8 k rows lost 3 % of a pass), the wide gathers
  // and the sweeps over the graph (their loads are ordered worse behind it: 2.4 M rows at 256 columns lost 20 %).
  template <typename... Args>
  void launch_alone(void (*kernel)(Args...), dim3 grid, int threads, size_t smem, typename Same<Args>::type... args) {
    joined = true;
    launch(kernel, grid, threads, smem, args...);
  }
  bool joined = false;   // the next launch takes the ordinary dependency
  bool in_pass = true;   // false: a propagation on its own
  void join(cudaStream_t waiting, cudaEvent_t e) {
    CU(cudaStreamWaitEvent(waiting, e, 0));
    joined = true;
  }

  // The propagation kernels on a graph given by its tables (the handle's own, or a rank's local part of it); x and
  // out have ldv vectors of VEC floats per row.
  template <int VEC, bool MAPPED, bool RELU = false>
  void spmm_tables(const GatherGraph& g, const float* xf, float* outf, int ldv, float* row_max = nullptr) {
    using T = typename gk::Vec<VEC>::T;
    const T* x = reinterpret_cast<const T*>(xf);
    T *out = reinterpret_cast<T*>(outf), *scratch = reinterpret_cast<T*>(g.item_sums);
    const int ld4 = (int)cdiv((long long)ldv * VEC, 4);
    const long long units = (long long)g.n + g.n_items;
    in_pass = !MAPPED;   // the caller's matrices: a call of its own
#define WIDE(NV4, UN, SLICED)                                                                                             \
  launch_alone(gk::k_spmm_wide<VEC, 4 / VEC * (NV4), UN, MAPPED, SLICED, RELU>, dim3((unsigned)cdiv(units * 32, 64), (unsigned)std::min<long long>(32768, cdiv(ld4, 32 * (NV4))),                \
              (unsigned)cdiv(ld4, 32768LL * 32 * (NV4))), 64, 0,                                                \
      g.row_ptr, g.col, g.dinv, g.perm, g.items, g.n, g.n_items, g.long_len, x, out, ldv, scratch, row_max)
#define SETS(CL, EP, UN) SETS_OF(1, CL, EP, UN)
#define SETS_OF(NV4, CL, EP, UN)                                                                                          \
  launch(gk::k_spmm_sets<VEC, 4 / VEC * (NV4), CL, EP, UN, MAPPED, RELU>, (unsigned)cdiv(units * ((CL) * (EP)), 128), 128, 0,  \
      g.row_ptr, g.col, g.dinv, g.perm, g.user_col, g.items, g.n, g.n_items, g.long_len, x, out, ldv, scratch, g.row_table, gk::ItemRows{g.rows, g.item_row, g.row_done}, row_max)
    // Sets of entries per row: as many as the warp holds while the grid is then still small (latency counts), fewer
    // where the rows alone fill the chip several times over and the lanes of half-empty sets would only cost issue
    // slots.  Lines between the measured sizes 0.2 / 1.4 / 20 M lanes (columns x rows); the rule reads the handle's n, so a
    // rank's part of a graph is summed in the order of the whole.
    const long long lanes = n * (ld4 <= 1 ? 1 : ld4 <= 2 ? 2 : ld4 <= 4 ? 4 : ld4 <= 8 ? 8 : 16);
    if (ld4 <= 1) {
      if (lanes <= 60000) SETS(1, 16, 4); else if (lanes <= 500000) SETS(1, 8, 4); else SETS(1, 4, 4);
    } else if (ld4 <= 2) {
      if (lanes <= 120000) SETS(2, 8, 4); else if (lanes <= 1000000) SETS(2, 4, 4); else SETS(2, 2, 4);
    } else if (ld4 <= 4) {
      if (lanes <= 240000) SETS(4, 8, 4); else SETS(4, 2, 4);
    } else if (ld4 <= 8) {
      if (VEC == 4 && lanes <= 160000) SETS_OF(2, 4, 4, 4); else if (lanes <= 480000) SETS(8, 4, 8); else SETS(8, 1, 8);
    } else if (VEC == 4 && ld4 <= 12) {
      // four lanes of three vectors leave none idle (us, against 16 lanes: 76 -> 65 at 169 k rows, 2469 -> 2115 at 2.45 M); of twelve
      // single floats, for a matrix of odd width, they are slower.  As many sets as there: all layouts of a width agree bit for bit.
      if (lanes <= 960000) SETS_OF(3, 4, 2, 4); else SETS_OF(3, 4, 1, 4);
    } else if (ld4 <= 16) {
      if (lanes <= 960000) SETS(16, 2, 8); else SETS(16, 1, 8);
    } else if (ld4 <= 32) WIDE(1, 4, false);
    else if (ld4 > 64) WIDE(2, 2, true);
    else WIDE(2, 2, false);   // two neighbours in flight per lane beat four (fewer registers, more warps): measured
#undef WIDE
#undef SETS
#undef SETS_OF
    in_pass = true;
    CU(cudaGetLastError());
    if (ld4 > 16 && g.n_long > 0) {
      launch(gk::k_spmm_long_rows<T, MAPPED>, (unsigned)g.n_long, 64, 0, g.rows, scratch, out, ldv, g.perm, row_max);
      CU(cudaGetLastError());
      ++launches;   // booked with the propagation it completes
    }
  }

  // Whether C = A B with these sizes runs on the tensor cores (K capped at 2048 because the accumulator error grows with K,
  // about 2.5e-9 K of the magnitude), and how: columns per group, and whether by split halves (B then comes as an image).
  bool on_tensor_cores(long long Mr, int K) const { return p.tensor_cores && K >= 8 && K <= 2048 && Mr >= 512; }
  static int group_width(int N, bool halves) {
    return N <= 16 ? 16 : N <= 32 ? 32 : N <= 48 ? 48 : N <= 64 ? 64 : halves && N <= 96 ? 96 : N <= 128 ? 128 : halves && N <= 192 ? 192 : 256;
  }
  // With many row tiles k_gemm_tc_ws would split the same weights again for every tile; with at most one tile per CTA, or
  // with few chunks, that costs nothing, and the image would (13.8 k rows, 767 x 1000, three tiles per CTA:
  // 130 -> 98 us by an image; 10 x 1000: no gain).
  bool by_halves(long long Mr, int N, int K) const {
    if (!on_tensor_cores(Mr, K) || encode_tiled() == nullptr) return false;
    return p.tensor_cores == 2 || Mr >= kHalfMinRows || (K >= 128 && cdiv(Mr, gtc::kBlockM) > kSmCount / cdiv(N, group_width(N, true)));
  }
  static size_t image_bytes(int N, const gtc::Image& im) {
    const int groups = (int)cdiv(N, im.nt);
    return gtc::image_blocks_bytes(groups, im.nt, im.kc) + (size_t)groups * im.nt * sizeof(float) + (size_t)gtc::image_marks(groups, im.nt, im.kc) * sizeof(int);
  }
  // Asks for an image of the operand of an n x K by K x N product, where that product takes one.
  void want_image(gtc::Image& im, int N, int K) {
    im = gtc::Image{nullptr, group_width(N, true), (int)cdiv(K, gtc::kChunkK)};
    if (by_halves(n, N, K)) want(im.data, image_bytes(N, im), kZero);
  }
  void split_b(const gtc::SplitB& b) {
    const int rows = (int)(cdiv(b.N, b.image.nt) * b.image.nt);
    Scope sc(this, "split_b", 1, 8.0 * (double)b.N * b.K, 0.0);
    launch(gtc::k_split_b, (unsigned)cdiv(rows, gtc::kSplitColumns), 256, 0, b, rows);
    CU(cudaGetLastError());
  }

  // C = A B.  B is handed over twice: row-major K x N (ldb) for the fp32-ALU kernels and K-major N x K (Bk, ldbk; may be
  // NULL) for the tensor-core kernels, which are used whenever they apply; a_max, image: the row maxima of A and the image of B,
  // for the product by split halves.
  void gemm_nn(const float* A, int lda, const float* a_max, const float* B, int ldb, const float* Bk, int ldbk, float* Cm, int ldc,
               long long Mr, int N, int K, const gtc::Image& image, const int* skip = nullptr) {
    char name[48];
    if (Bk != nullptr && on_tensor_cores(Mr, K)) {
      CUtensorMap tmap;
      const bool halves = by_halves(Mr, N, K) && a_max != nullptr && image.data != nullptr && make_a_tile_map(A, Mr, lda, &tmap);
      const int tiles = (int)cdiv(Mr, gtc::kBlockM), nt = group_width(N, halves), groups = (int)cdiv(N, nt), kc = (int)cdiv(K, gtc::kChunkK);
      std::snprintf(name, sizeof name, halves ? "gemm_half@%dx%d" : "gemm_tc@%dx%d", K, N);
      Scope sc(this, name, 1, 4.0 * ((double)Mr * (lda + ldc) + (double)K * ldb), 2.0 * (double)Mr * N * K);
      dim3 grid((unsigned)std::max(1, std::min(tiles, kSmCount / groups)), (unsigned)groups);
      // few row tiles and a long reduction: several CTAs share a tile's K chunks, at least four chunks each
      // (2.7 k rows, K = 1433, 16 columns: 34 -> 13 us)
      if (!halves)
        grid.z = (unsigned)std::max<long long>(1, std::min<long long>({kSmCount / ((long long)tiles * groups), kc / 4,
                                                                       (long long)(part_elems / ((size_t)Mr * ldc))}));
      auto with_width = [&](auto width) {
        constexpr int NT = decltype(width)::value;
        if (halves) {
          using Cfg = gtc::HalfCfg<NT>;
          CU(cudaFuncSetAttribute(gtc::k_gemm_half<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem));
          launch_alone(gtc::k_gemm_half<NT>, grid, Cfg::kThreads, Cfg::kSmem, A, lda, a_max, Bk, ldbk, Cm, ldc, (int)Mr, N, K, skip, tc_error, image.data, tmap);
        } else if constexpr (NT != 96 && NT != 192) {
          using Cfg = gtc::WsCfg<NT>;
          CU(cudaFuncSetAttribute(gtc::k_gemm_tc_ws<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem));
          launch_alone(gtc::k_gemm_tc_ws<NT>, grid, Cfg::kThreads, Cfg::kSmem, A, lda, Bk, ldbk, Cm, ldc, (int)Mr, N, K, skip, tc_error, part, tile_tickets);
        }
      };
      switch (nt) {
        case 16: with_width(std::integral_constant<int, 16>()); break;
        case 32: with_width(std::integral_constant<int, 32>()); break;
        case 48: with_width(std::integral_constant<int, 48>()); break;
        case 64: with_width(std::integral_constant<int, 64>()); break;
        case 96: with_width(std::integral_constant<int, 96>()); break;
        case 128: with_width(std::integral_constant<int, 128>()); break;
        case 192: with_width(std::integral_constant<int, 192>()); break;
        default: with_width(std::integral_constant<int, 256>());
      }
      CU(cudaGetLastError());
      return;
    }
    std::snprintf(name, sizeof name, "gemm_nn@%dx%d", K, N);
    Scope sc(this, name, 1, 4.0 * ((double)Mr * (lda + ldc) + (double)K * ldb), 2.0 * (double)Mr * N * K);
#define NN_CASE(BM, BN, BK, TM, TN)                                                             \
  {                                                                                             \
    dim3 grid((unsigned)cdiv(Mr, BM), (unsigned)cdiv(ldc, BN));                                  \
    launch_alone(gk::k_gemm_nn<BM, BN, BK, TM, TN>, grid, (BM / TM) * (BN / TN), 0, A, lda, B, ldb, Cm, ldc, (int)Mr, N, K, skip); \
  }
    if (N > 64) NN_CASE(128, 128, 16, 8, 8)
    else if (N > 16) NN_CASE(128, 64, 16, 8, 4)
    else NN_CASE(256, 16, 16, 4, 4)
#undef NN_CASE
    CU(cudaGetLastError());
  }

  // A^T B over `rows` rows as split partial sums in `part` (added up in a fixed order by finish_grad); returns their number.
  // Whether P^T R runs on the tensor cores (that form can also build a hidden layer's R itself).
  bool tn_on_tensor_cores(long long rows) const { return p.tensor_cores != 0 && rows >= 4096; }

  // With `zres` B holds pre-activations H and the operand is
  // h > 0 ? nu (h - z) : 0, formed while staging: the residual matrix is never stored.
  int gemm_tn(const float* A, int lda, const float* B, int ldb, int ldp, long long rows, int Ka, int Nb,
              const float* zres = nullptr, float nu = 0.f) {
    int splits = 1;
    long long rps = rows;
    char name[48];
    if (tn_on_tensor_cores(rows)) {
      std::snprintf(name, sizeof name, zres ? "gemm_tn_tc.resid@%dx%d" : "gemm_tn_tc@%dx%d", Ka, Nb);
      Scope sc(this, name, 1, 4.0 * ((double)rows * (lda + (zres ? 2 : 1) * ldb) + (double)Ka * ldp), 2.0 * (double)rows * Ka * Nb);
      const int nt_tn = Nb <= 16 ? 16 : Nb <= 32 ? 32 : Nb <= 48 ? 48 : Nb <= 64 ? 64 : Nb <= 128 ? 128 : 256;
      const int nb_groups = (int)cdiv(Nb, nt_tn);
      const int groups = (int)cdiv(Ka, gtc::kBlockM);
      // at most 2048 rows (256 MMAs) per accumulator: the tensor core rounds the running sum toward zero at
      // every MMA, so long sums are cut into splits whose partial results are added in fp64
      splits = (int)std::max<long long>(std::max(1, kSmCount / (groups * nb_groups)), cdiv(rows, 2048));
      {   // whole waves: with more CTAs than SMs (one CTA per SM), round the count up to a multiple of the SM count
        const long long per = (long long)groups * nb_groups;
        if (splits * per > kSmCount) splits = (int)(cdiv(splits * per, kSmCount) * kSmCount / per);
      }
      splits = (int)std::min<long long>(splits, cdiv(rows, 256));
      splits = (int)std::min<long long>(splits, (long long)(part_elems / ((size_t)Ka * ldp)));
      rps = cdiv(rows, splits);
      splits = (int)cdiv(rows, rps);
#define TN_TC(NT)                                                                                              \
  {                                                                                                            \
    const size_t smem = zres ? gtc::TnCfg<NT, true>::kSmem : gtc::TnCfg<NT, false>::kSmem;                     \
    dim3 grid((unsigned)groups, (unsigned)splits, (unsigned)nb_groups);                                        \
    if (zres) {                                                                                                \
      CU(cudaFuncSetAttribute(gtc::k_gemm_tn_tc<NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
      launch_alone(gtc::k_gemm_tn_tc<NT, true>, grid, gtc::kTnThreads, smem, A, lda, B, ldb, part, ldp, rows, rps, Ka, Nb, tc_error, zres, nu); \
    } else {                                                                                                   \
      CU(cudaFuncSetAttribute(gtc::k_gemm_tn_tc<NT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
      launch_alone(gtc::k_gemm_tn_tc<NT, false>, grid, gtc::kTnThreads, smem, A, lda, B, ldb, part, ldp, rows, rps, Ka, Nb, tc_error, nullptr, 0.f); \
    }                                                                                                          \
  }
      if (Nb <= 16) TN_TC(16)
      else if (Nb <= 32) TN_TC(32)
      else if (Nb <= 48) TN_TC(48)
      else if (Nb <= 64) TN_TC(64)
      else if (Nb <= 128) TN_TC(128)
      else TN_TC(256)
#undef TN_TC
      CU(cudaGetLastError());
      return splits;
    }
    std::snprintf(name, sizeof name, zres ? "gemm_tn.resid@%dx%d" : "gemm_tn@%dx%d", Ka, Nb);
    Scope sc(this, name, 1, 4.0 * ((double)rows * (lda + (zres ? 2 : 1) * ldb) + (double)Ka * ldp), 2.0 * (double)rows * Ka * Nb);
#define TN_CASE(BM, BN, BK, TM, TN)                                                             \
  {                                                                                             \
    const long long tiles = cdiv(Ka, BM) * cdiv(ldp, BN);                                        \
    splits = (int)std::max<long long>(1, std::min<long long>((4LL * kSmCount) / tiles, cdiv(rows, 64))); \
    splits = (int)std::min<long long>(splits, (long long)(part_elems / ((size_t)Ka * ldp)));     \
    rps = cdiv(rows, splits);                                                                    \
    splits = (int)cdiv(rows, rps);                                                               \
    dim3 grid((unsigned)cdiv(Ka, BM), (unsigned)cdiv(ldp, BN), (unsigned)splits);                \
    if (zres) launch_alone(gk::k_gemm_tn<BM, BN, BK, TM, TN, true>, grid, (BM / TM) * (BN / TN), 0, A, lda, B, ldb, part, ldp, rows, rps, Ka, Nb, zres, nu); \
    else launch_alone(gk::k_gemm_tn<BM, BN, BK, TM, TN, false>, grid, (BM / TM) * (BN / TN), 0, A, lda, B, ldb, part, ldp, rows, rps, Ka, Nb, nullptr, 0.f); \
  }
    if (Nb > 64) TN_CASE(128, 128, 16, 8, 8)
    else if (Nb > 16) TN_CASE(128, 64, 16, 8, 4)
    else if (Nb > 8) TN_CASE(128, 16, 16, 8, 1)
    else TN_CASE(128, 8, 16, 4, 1)
#undef TN_CASE
    CU(cudaGetLastError());
    return splits;
  }

  // grad (and grad_t) from the `splits` partial sums gemm_tn left in `part`; with `ctl` the start of the W_l search too.
  void finish_grad(int splits, int Ka, int Nb, int ldp, float* out, float* out_t, int ldt, const float* w, SearchCtl* ctl,
                   bool maxima) {
    Scope sc(this, "finish_grad", 1, 4.0 * (double)Ka * ldp * (splits + (w ? 3 : 1)), 0.0);
    const long long elems = (long long)Ka * ldp;
    if (splits >= 16)
      launch(gk::k_finish_grad<8>, (unsigned)cdiv(elems, 32), 256, 0, part, splits, Ka, Nb, ldp, out, out_t, ldt, w, red_part,
                                                                            ticket, ctl, p.bt_shrink, p.bt_growth, status, maxima);
    else
      launch(gk::k_finish_grad<1>, (unsigned)(cdiv(Ka, 32) * cdiv(ldp, 32)), 256, 0, part, splits, Ka, Nb, ldp, out, out_t, ldt, w, red_part,
                                                                                     ticket, ctl, p.bt_shrink, p.bt_growth, status, maxima);
    CU(cudaGetLastError());
  }

  // Blocks of `kernel` that fit the device at once (looked up once per kernel and shared-memory size): the grid of a
  // cooperative or persistent launch.
  std::map<std::pair<const void*, size_t>, int> resident_cache;
  int resident_blocks(const void* kernel, int threads, size_t smem) {
    auto it = resident_cache.find({kernel, smem});
    if (it != resident_cache.end()) return it->second;
    allow_shared(p.device, kernel, smem);
    int per_sm = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
    if (per_sm < 1) throw Fail{GCN_ADMM_ERR_CUDA, "a kernel does not fit the device"};
    return resident_cache[{kernel, smem}] = per_sm * kSmCount;
  }
  template <typename... Args>
  void launch_together(void (*kernel)(Args...), long long blocks_wanted, int threads, size_t smem, typename Same<Args>::type... args) {
    const void* f = reinterpret_cast<const void*>(kernel);
    const int grid = (int)std::max<long long>(1, std::min<long long>(blocks_wanted, resident_blocks(f, threads, smem)));
    void* argv[] = {const_cast<void*>(static_cast<const void*>(&args))...};
    CU(cudaLaunchCooperativeKernel(f, dim3((unsigned)grid), dim3((unsigned)threads), argv, smem, stream));
  }

  void resid(int l, float* R) {   // derivative of phi_l with respect to H_l, at the stored H_l
    const long long n4 = n * ld[l] / 4;
    Scope sc(this, l < L ? "resid_hidden" : "resid_out", 1, 16.0 * n4 * (l < L ? 3 : 4), 0.0);
    if (l < L)
      launch(gk::k_resid_hidden, grid_for(n4), 256, 0, (const float4*)H[l], (const float4*)Z[l], (float4*)R, n4, p.nu);
    else
      launch(gk::k_resid_out, grid_for(n4), 256, 0, (const float4*)H[l], (const float4*)Z[l], (const float4*)U,
                                                        (float4*)R, n4, p.rho);
    CU(cudaGetLastError());
  }

  long long z_per_pass() const { return (long long)std::max(L - 1, 0) * M; }
  gk::DecisionLog log_w(int l) const { return gk::DecisionLog{log_trial_w, log_q_w, d_pass, L, l - 1, kLogPasses}; }
  gk::DecisionLog log_z(int l) const {
    return gk::DecisionLog{log_trial_z, log_q_z, d_pass, z_per_pass(), (long long)(l - 1) * M, kLogPasses};
  }

  // A single block family is about to run: everything else is logged as "not run".
  void clear_log_pass() {
    const long long zc = z_per_pass();
    Scope sc(this, "small", zc > 0 ? 2 : 1, 0.0, 0.0);
    gk::k_log_clear<<<1, 64, 0, stream>>>(log_trial_w, d_pass, L, kLogPasses);
    if (zc > 0) gk::k_log_clear<<<grid_for(zc), 256, 0, stream>>>(log_trial_z, d_pass, zc, kLogPasses);
    CU(cudaGetLastError());
  }

  // ---- W_l block (Section 3.1) --------------------------------------------------------
  // Where R_l is formed and, turned into its value at the new H_l, handed from the W_l update to that of Z_{l-1}.
  float* resid_of(int l) const { return l == L && RL != nullptr ? RL : B0; }
  // resid_next: also leave the derivative of phi_l at the new H_l in resid_of(l) (what the Z_{l-1} update starts from).
  void update_W(int l, bool resid_next) {
    Range range("gcn_admm: W block");
    const int Kp = C[l - 1], Cn = C[l], ldc = ld[l];
    const long long n4 = n * ldc / 4;
    SearchCtl* ctl = ctl_w + l;
    float *const R = resid_of(l), *const D = l == L && DL != nullptr ? DL : B1;
    int splits;
    if (l < L) {                                                        // grad = P_l^T R_l, R_l formed inside the product
      splits = gemm_tn(P[l], ld[l - 1], H[l], ldc, ldc, n, Kp, Cn, Z[l], p.nu);
    } else {
      resid(l, R);                                                      // R_l
      splits = gemm_tn(P[l], ld[l - 1], R, ldc, ldc, n, Kp, Cn);   // grad = P_l^T R_l
    }
    finish_grad(splits, Kp, Cn, ldc, grad, grad_t, ld[l - 1], W[l], ctl, img_H[l].data != nullptr || img_G[l].data != nullptr);
    // in a launch of its own, for the scales: only a finished gradient gives each column its largest element
    if (img_D[l].data != nullptr) split_b(gtc::SplitB{grad_t, ld[l - 1], Cn, Kp, img_D[l]});
    gemm_nn(P[l], ld[l - 1], P_max[l], grad, ldc, grad_t, ld[l - 1], D, ldc, n, Cn, Kp, img_D[l], &ctl->done);   // D = P_l grad
    gk::SearchW a{};
    a.H = (float4*)H[l]; a.D = (const float4*)D; a.Z = (const float4*)Z[l]; a.U = (const float4*)U; a.R = (const float4*)R;
    a.Rn = resid_next ? (float4*)R : nullptr;
    a.n4 = n4;
    a.coef = l == L ? p.rho : p.nu;
    a.W = W[l]; a.Wt = Wt[l]; a.image = img_H[l]; a.image_t = img_G[l]; a.grad = grad;
    a.rows = Kp; a.cols = Cn; a.ldw = ldc; a.ldwt = ld[l - 1];
    a.ctl = ctl; a.partial = red_part; a.bar = grid_bar; a.ticket = ticket; a.status = status; a.err = tc_error;
    a.a.growth = p.bt_growth;
    a.a.max_trials = p.bt_max_trials;
    a.a.cand = gk::kCand;
    a.a.mode = l == L ? 1 : 0;
    a.a.scale = 0.5 * p.nu;
    a.a.quad_coef = 0.5 * p.rho;
    a.log = log_w(l);
    // the move reads two arrays and writes one; the next residual reads one more (two for the last layer) and writes one
    if (l == L) {
      {
        Scope sc(this, "score_w_out", 1, 32.0 * n4, 0.0);
        launch(gk::k_score_w_out, grid_for(n4), 256, 0, a);
        CU(cudaGetLastError());
      }
      {
        Scope sc(this, "move_w_out", 1, 16.0 * (3 + (resid_next ? 3 : 0)) * n4, 0.0);
        launch(gk::k_move_w_out, grid_for(n4), 256, 0, a);
        CU(cudaGetLastError());
      }
    } else {
      Scope sc(this, "search_w_hidden", 1, 16.0 * (6 + (resid_next ? 2 : 0)) * n4, 0.0);
      launch_together(gk::k_search_w_hidden, cdiv(n4, 256), 256, 0, a);
    }
  }

  // Whether the update of Z_l forms its gradient and T in one launch (k_zgrad_products).  What it saves is launches and passes of G
  // through memory, what it costs is the rate of fp32 FMA out of shared memory, so the line lies by the next layer's width against
  // this one's and by n.  us a pass, separate / joined: 64-128-4 at 4 k, 170 k and 600 k rows 110 / 101, 657 / 602, 2024 / 1927;
  // 64-256-16 149 / 139, 1124 / 1102, 3700 / 3596; 64-128-16 112 / 102, 697 / 708, 2156 / 2274; 64-32-8 84 / 75, 346 / 351, 1009 / 1048;
  // 64-64-31 at 1 k, 4 k, 8 k, 16 k 75 / 69, 92 / 85, 100 / 98, 132 / 138; 64-64-47 78 / 74, 97 / 91, 107 / 112, 142 / 162.
  bool joins_products(int l) const {
    const long long ldl = ld[l], ldn = ld[l + 1];
    if (ldn > 48 || (ldn + 12) * ldl * sizeof(float) > 96 * 1024) return false;
    if (ldn > 16) return n <= (ldn <= 32 ? 8192 : 4096);
    return n <= 65536 || ldn <= 4 || ldl >= 16 * ldn;
  }

  // ---- Z_{l,m}, l < L, every community (Appendix A, Eq. 5/6 and 8-10) ------------------
  // resid_ready: resid_of(l + 1) holds the derivative of phi_{l+1} at the stored H_{l+1}.
  void update_Z_hidden(int l, bool resid_ready) {
    Range range("gcn_admm: hidden Z blocks");
    const int ldl = ld[l], ldn = ld[l + 1];
    SearchCtl* ctl = ctl_z + (size_t)l * M;
    float* const Rn = resid_of(l + 1);
    if (!resid_ready) resid(l + 1, Rn);                                  // R'_{l+1}
    spmm(Rn, B1, ldn, !joins_products(l) && img_G[l + 1].data != nullptr ? B1_max : nullptr);                      // S = A~ R'
    // G = S W_{l+1}^T + nu (Z_l - f(H_l)) and T = G W_{l+1}: in one launch where the next layer is narrow (see k_zgrad_products)
    const bool joined = joins_products(l);
    if (joined) {
      Scope sc(this, "zgrad_products", 1, 4.0 * (double)n * (3.0 * ldl + 2.0 * ldn), 4.0 * (double)n * C[l] * C[l + 1]);
      const auto finish = [&](auto kernel, int kv, int rows) {
        static_assert(kZBlockRows == 32, "a block's groups of eight lanes take 32 rows");
        const size_t smem = (size_t)kv * 4 * ldl * sizeof(float);
        const int blocks = std::min(n_zblocks, resident_blocks((const void*)kernel, 256 / rows, smem));
        launch(kernel, (unsigned)blocks, 256 / rows, smem, (float4*)B2, (const float4*)Z[l], (const float4*)H[l], (const float4*)B1, (const float4*)Wt[l + 1], (float4*)B0,
               ldl / 4, C[l + 1], d_zblocks, n_zblocks, p.nu, red_part, d_comm_block_ptr, comm_tickets, ctl, sums_z, p.bt_shrink, p.bt_growth, n_active, status);
      };
      if (ldn <= 4) finish(gk::k_zgrad_products<1, 2>, 1, 2);
      else if (ldn <= 8) finish(gk::k_zgrad_products<2, 2>, 2, 2);
      else if (ldn <= 12) finish(gk::k_zgrad_products<3, 2>, 3, 2);
      else if (ldn <= 16) finish(gk::k_zgrad_products<4, 2>, 4, 2);
      else if (ldn <= 24) finish(gk::k_zgrad_products<6, 1>, 6, 1);
      else if (ldn <= 32) finish(gk::k_zgrad_products<8, 1>, 8, 1);
      else finish(gk::k_zgrad_products<12, 1>, 12, 1);
      CU(cudaGetLastError());
    } else {
      gemm_nn(B1, ldn, B1_max, Wt[l + 1], ldl, W[l + 1], ldn, B2, ldl, n, C[l], C[l + 1], img_G[l + 1]);
      Scope sc(this, "zgrad_finish", 1, 16.0 * 4.0 * (double)n * (ldl / 4), 0.0);
      const auto finish = [&](auto kernel) {
        launch(kernel, (unsigned)n_zblocks, 256, 0, (float4*)B2, (const float4*)Z[l], (const float4*)H[l], ldl / 4, d_zblocks, p.nu, red_part, d_comm_block_ptr, comm_tickets, ctl, sums_z,
               p.bt_shrink, p.bt_growth, n_active, status, img_H[l + 1].data != nullptr ? B2_max : nullptr);
      };
      if (ldl <= 16) finish(gk::k_zgrad_finish<4>);
      else finish(gk::k_zgrad_finish<8>);   // whole lines still, and few idle lanes at any width
      CU(cudaGetLastError());
    }
    const int ld4 = ldn / 4, warps = 8;
    const double move_bytes = 12.0 * (double)n * ldl;
    char zname[48];
    float4* const scratch = reinterpret_cast<float4*>(item_sums);
    gk::DecideArgs decide{};
    decide.growth = p.bt_growth;
    decide.max_trials = p.bt_max_trials;
    decide.own_nu = p.nu;
    if (l + 1 == L) {   // closed form
      if (!joined) gemm_nn(B2, ldl, B2_max, W[L], ldn, Wt[L], ldl, B0, ldn, n, C[L], C[l], img_H[L]);   // T = G W_L; S stays in B1
      decide.mode = 1;
      decide.quad_coef = 0.5 * p.rho;
      gk::SearchOut a{};
      a.segs = d_segs; a.chunks = d_seg_chunks; a.n_chunks = n_seg_chunks; a.chunk_counter = chunk_counter;
      a.slot_ptr = d_slot_ptr; a.slots = slots; a.comm_done = comm_done; a.split_done = split_done; a.items = d_items; a.split = d_split;
      a.ctl = ctl; a.own = sums_z; a.n_active = n_active; a.status = status; a.a = decide;
      // The longest segments are the critical path.  A warp shared by 32 / CL sets walks one in as many fewer steps, a short one in
      // none fewer but with its sets half empty, so the line lies the higher the fewer sets there are.  us at 6 / 24 / 48 / 128 /
      // never: 3 columns (19.7 k rows, 2 entries each) 21.0 / 20.8 / 21.5 / 22.6 / 22.5, 10 (13.8 k, 30) 36.9 / 35.1 / 36.6 / 41.2 /
      // 52.2, 4 (600 k, 40) 456 / 314 / 305 / 304 / 305; 23 (30 k, 16) 34.2 / 32.2 / 32.9 / 35.4 / 44.6, 23 (20 k, 50) 47.1 / 41.2 /
      // 40.8 / 43.3 / 51.6; 40 (169 k, 14) 113 / 104 / 103 / 103 / 105, 47 (600 k, 50) 1032 / 934 / 915 / 899 / 896, 47 (2.45 M, 51)
      // 4181 / 3850 / 3771 / 3743 / 3756.  With CL = 32 there is one set and no difference.
      a.share_from = ld4 <= 4 ? 24 : ld4 <= 8 ? 48 : 128;
      std::snprintf(zname, sizeof zname, "search_z_out@%d", ldn);
      {
        Scope sc(this, zname, 1, 4.0 * gi.nnz + 12.0 * n + 8.0 * (double)n * ldn, 2.0 * (double)gi.nnz * ldn);
        const auto search = [&](auto kernel, int grid, int block) {
          launch_alone(kernel, grid, block, 0, d_col, d_dinv, (const float4*)B0, (const float4*)B1, ld4, scratch, a);
        };
        const int dealt = (int)cdiv(n_seg_chunks, 2);
#define NARROW(CL)                                                                                     \
  {                                                                                                    \
    const int grid = resident_blocks((const void*)gk::k_search_z_out<CL, false>, warps * 32, 0);       \
    if (n_seg_chunks <= grid * warps) search(gk::k_search_z_out<CL, true>, dealt, 64);                 \
    else search(gk::k_search_z_out<CL, false>, grid, warps * 32);                                      \
  }
        if (ld4 <= 1) NARROW(1)
        else if (ld4 <= 2) NARROW(2)
        else if (ld4 <= 4) NARROW(4)
        else if (ld4 <= 8) search(gk::k_search_z_out<8, true>, dealt, 64);
        else if (ld4 <= 16) search(gk::k_search_z_out<16, true>, dealt, 64);
        else search(gk::k_search_z_out<32, true>, dealt, 64);
#undef NARROW
        CU(cudaGetLastError());
      }
      Scope sc(this, "move_z", 1, move_bytes, 0.0);
      launch(gk::k_move_z, grid_for(n * (ldl / 4)), 256, 0, (float4*)Z[l], (const float4*)B2, ldl / 4, n, d_row_comm, ctl, M, log_z(l),
                                                                chunk_counter);
      CU(cudaGetLastError());
      return;
    }
    if (!joined) gemm_nn(B2, ldl, B2_max, W[l + 1], ldn, Wt[l + 1], ldl, B0, ldn, n, C[l + 1], C[l], img_H[l + 1]);   // T = G W_{l+1}
    decide.cand = gk::kCand;   // steady-state searches close at trial 0..2
    decide.scale = 0.5 * p.nu;
    gk::SearchZ a{};
    a.ctl = ctl; a.n_comm = M;
    a.chunk_part = z_chunk_part; a.chunk_counter = chunk_counter; a.group_part = z_group_part;
    // few chunks: a warp per community adds them up directly; many: group by group first (one more meeting of the grid)
    a.per_group = (int)cdiv(n_chunks, kChunkGroups);
    a.n_groups = n_chunks > kChunkGroups ? (int)cdiv(n_chunks, a.per_group) : 0;
    a.split = d_split; a.n_split = n_split; a.split_scores = split_scores; a.split_order = d_split_order; a.split_ptr = d_split_ptr;
    a.own = sums_z; a.n_active = n_active; a.status = status; a.err = tc_error; a.bar = grid_bar;
    a.a = decide;
    a.log = log_z(l);
    a.Z = (float4*)Z[l]; a.G = (const float4*)B2; a.ldz4 = ldl / 4; a.row_comm = d_row_comm;
    std::snprintf(zname, sizeof zname, "score_z_hidden@%d", ldn);
    const float4 *T = (const float4*)B0, *Hn = (const float4*)H[l + 1], *Zn = (const float4*)Z[l + 1];
    const size_t sums = (size_t)warps * M * gk::kCand * sizeof(double);
    const int use_smem = sums <= 96 * 1024;
    auto score = [&](auto kernel, auto close, int V) {
      const size_t smem = (size_t)warps * 2 * V * 32 * sizeof(float4) + (use_smem ? sums + (size_t)M * sizeof(float4) : 0);
      const int grid = (int)std::min<long long>(cdiv(n_chunks, warps), resident_blocks((const void*)kernel, warps * 32, smem));
      {
        Scope sc(this, zname, 1, 6.0 * gi.nnz + 8.0 * n + 12.0 * (double)n * ldn, 2.0 * (double)gi.nnz * ldn);
        launch_alone(kernel, grid, warps * 32, smem, d_row_ptr, d_col, d_col_comm, d_dinv, T, Hn, Zn, ld4, ctl, M, z_chunk_part, n_active,
               use_smem, d_chunk_ptr, n_chunks, chunk_counter, d_items, n_items, long_len, scratch);
        CU(cudaGetLastError());
      }
      // closing, further sweeps and the move: as many blocks as the move can use
      Scope sc(this, "close_z", 1, move_bytes, 0.0);
      launch_together(close, cdiv(n * (ldl / 4), 256), warps * 32, smem, d_row_ptr, d_col, d_col_comm, d_dinv, T, Hn, Zn, ld4, (int)n,
                      use_smem, d_chunk_ptr, n_chunks, d_items, n_items, long_len, scratch, a);
    };
    if (ld4 <= 32) score(gk::k_score_z<1, 4>, gk::k_close_z<1, 4>, 1);
    else if (ld4 <= 64) score(gk::k_score_z<2, 4>, gk::k_close_z<2, 4>, 2);
    else if (ld4 <= 128) score(gk::k_score_z<4, 4>, gk::k_close_z<4, 4>, 4);
    else score(gk::k_score_z<8, 4>, gk::k_close_z<8, 4>, 8);
  }

  // ---- Z_L (Eq. 7) and, in the same sweep, the dual as printed in Eq. 3 -----------------
  void update_output(bool dual_now, bool update_z) {
    Range range("gcn_admm: output layer and dual");
    Scope sc(this, "output_rows", 1, 4.0 * (double)n * ld[L] * (3 + (update_z ? 1 : 0) + (dual_now ? 1 : 0)), 0.0);
    gk::OutputArgs a{};
    a.Z = Z[L]; a.U = U; a.H = H[L];
    a.ld = ld[L]; a.C = C[L]; a.n = n;
    a.train = d_train; a.rows = d_train_rows; a.y = d_y; a.n_train = n_train; a.momentum = d_fista_momentum;
    a.rho = p.rho; a.loss_scale = p.loss_scale; a.iters = p.fista_iters;
    a.dual_now = dual_now ? 1 : 0; a.update_z = update_z ? 1 : 0;
    const int plain_blocks = grid_for(n * (ld[L] / 4));
#define OUTPUT(LPR, CPL)                                                        \
  {                                                                             \
    a.train_blocks = (int)cdiv((long long)n_train * (LPR), 256);                \
    launch(gk::k_output<LPR, CPL>, (unsigned)(a.train_blocks + plain_blocks), 256, 0, a); \
  }
    if (C[L] <= 4) OUTPUT(4, 1)
    else if (C[L] <= 8) OUTPUT(4, 2)
    else if (C[L] <= 16) OUTPUT(8, 2)
    else if (C[L] <= 24) OUTPUT(8, 3)
    else if (C[L] <= 32) OUTPUT(8, 4)
    else if (C[L] <= 40) OUTPUT(8, 5)
    else if (C[L] <= 48) OUTPUT(8, 6)
    else if (C[L] <= 64) OUTPUT(8, 8)
    else if (C[L] <= 96) OUTPUT(16, 6)
    else OUTPUT(16, 8)
#undef OUTPUT
    CU(cudaGetLastError());
  }

  void dual_from_stored() {   // U + rho (Z_L - H_L) with H_L = A~ Z_{L-1} W_L of the stored iterates
    const long long n4 = n * ld[L] / 4;
    Scope sc(this, "dual", 1, 64.0 * n4, 0.0);
    launch(gk::k_dual, grid_for(n4), 256, 0, (float4*)U, (const float4*)Z[L], (const float4*)H[L], n4, p.rho);
    CU(cudaGetLastError());
  }

  // P_l = A~ Z_{l-1} (l >= 2; P_1 is constant) and H_l = P_l W_l from the stored W, Z.
  // keep_h1: the caller knows that H_1 already is P_1 W_1.  After a pass it is: P_1 never changes and
  // the W_1 step left H_1 - D/tau = P_1 (W_1 - grad/tau) behind, so the product is skipped; to keep
  // rounding from piling up over many passes it is still formed afresh every kH1RefreshEvery passes.
  // A recorded pass launches the product every time and lets the device decide (*skip_h1, kept by k_end_pass).
  static constexpr int kH1RefreshEvery = 16;
  int h1_age = 0;
  bool capturing = false;
  void refresh(bool keep_h1 = false) {
    Range range("gcn_admm: refresh P_l, H_l");
    for (int l = 2; l <= L; ++l) spmm(Z[l - 1], P[l], ld[l - 1], P_max[l]);
    refresh_H1(keep_h1);
    for (int l = 2; l <= L; ++l) refresh_H(l);
    fresh = true;
  }
  void refresh_H(int l, const int* skip = nullptr) {
    gemm_nn(P[l], ld[l - 1], P_max[l], W[l], ld[l], Wt[l], ld[l - 1], H[l], ld[l], n, C[l], C[l - 1], img_H[l], skip);
  }
  void refresh_H1(bool keep_h1) {
    const bool skip = keep_h1 && !capturing && h1_age + 1 < kH1RefreshEvery;
    h1_age = skip ? h1_age + 1 : 0;
    if (!skip) refresh_H(1, keep_h1 && capturing ? skip_h1 : nullptr);
  }
  void end_pass() {
    Scope sc(this, "small", 1, 0.0, 0.0);
    launch(gk::k_end_pass, 1, 1, 0, d_pass, d_h1_age, skip_h1, kH1RefreshEvery);
    CU(cudaGetLastError());
    ++log_count;
  }

  // The serial schedule of Section 4.1: the same block updates, one after the other in the order
  // W_1, Z_1, .., W_L, Z_L, U, each reading the latest value of every other block.
  void iterate_sequential() {
    if (!fresh) refresh();
    for (int l = 1; l <= L; ++l) {
      if (l >= 2) {   // Z_{l-1} has just moved: P_l and H_l follow it (H_{l+1} still matches the untouched Z_l)
        spmm(Z[l - 1], P[l], ld[l - 1], P_max[l]);
        refresh_H(l);
      }
      update_W(l, false);
      if (l < L) update_Z_hidden(l, false);
      else update_output(false, true);
    }
    refresh(true);
    dual_from_stored();
    end_pass();
  }

  // A second line of launches for what does not depend on the hidden layers: the W_L update and the output layer's rows read
  // iterate k only (Jacobi), so on a graph too small to fill the chip they run beside W_1 .. W_{L-1} and Z_1 .. Z_{L-1} instead
  // of between them.  It has a stream, the scratch of the products and sums, and matrices of the last layer's width of its own.
  struct Lane {
    cudaStream_t stream = nullptr;
    float *part = nullptr, *grad = nullptr, *grad_t = nullptr;
    size_t part_elems = 0;
    double* red_part = nullptr;
    unsigned *ticket = nullptr, *tile_tickets = nullptr;
    cudaEvent_t begun = nullptr, w_done = nullptr, out_done = nullptr, done = nullptr;
  } side;
  bool two_lanes = false;
  void swap_lane() {   // launches go to the other line until the next call
    std::swap(stream, side.stream);
    std::swap(part, side.part);
    std::swap(part_elems, side.part_elems);
    std::swap(grad, side.grad);
    std::swap(grad_t, side.grad_t);
    std::swap(red_part, side.red_part);
    std::swap(ticket, side.ticket);
    std::swap(tile_tickets, side.tile_tickets);
  }

  template <typename F>
  void on_side(F&& launches_there) {
    swap_lane();
    try {
      launches_there();
    } catch (...) {
      swap_lane();
      throw;
    }
    swap_lane();
  }

  // Algorithm 1, one pass.  Z_{l-1} follows W_l directly, so that one matrix carries R_l from one to the other whatever the depth:
  // the W updates after it read P (not yet formed again), H, Z and U of other layers, none of which it writes.
  void iterate() {
    if (p.schedule == 1) { iterate_sequential(); return; }
    if (!fresh) refresh();
    if (!two_lanes || profiling) {
      for (int l = 1; l <= L; ++l) {
        update_W(l, l >= 2);
        if (l >= 2) update_Z_hidden(l - 1, true);
      }
      update_output(p.dual_mode == 0, true);
      refresh(true);
    } else {
      CU(cudaEventRecord(side.begun, stream));
      join(side.stream, side.begun);
      on_side([&] {
        update_W(L, true);
        CU(cudaEventRecord(side.w_done, stream));
        update_output(p.dual_mode == 0, true);
        CU(cudaEventRecord(side.out_done, stream));
      });
      for (int l = 1; l < L; ++l) {
        update_W(l, l >= 2);
        if (l >= 2) update_Z_hidden(l - 1, true);
      }
      join(stream, side.w_done);
      update_Z_hidden(L - 1, true);
      CU(cudaEventRecord(side.begun, stream));
      join(side.stream, side.begun);
      on_side([&] {
        refresh_H1(true);
        end_pass();
        CU(cudaEventRecord(side.done, stream));
      });
      for (int l = 2; l <= L; ++l) spmm(Z[l - 1], P[l], ld[l - 1], P_max[l]);
      join(stream, side.out_done);   // its rows of H_L have been read
      for (int l = 2; l <= L; ++l) refresh_H(l);
      join(stream, side.done);
      if (p.dual_mode != 0) dual_from_stored();
      return;
    }
    if (p.dual_mode != 0) dual_from_stored();
    end_pass();
  }

  void relu(const float* x, float* out, int ldx, float* out_max = nullptr) {
    Scope sc(this, "relu", 1, 8.0 * (double)n * ldx, 0.0);
    gk::k_relu<<<grid_for(32 * n), 256, 0, stream>>>((const float4*)x, (float4*)out, ldx / 4, n, out_max);
    CU(cudaGetLastError());
  }

  // Logits of Problem 1's forward pass with the stored W (N x ld_L, in H_1, B0 or B1; B2 is free).  The first layer's product
  // is H_1 itself while the stored matrices agree.  A (f(H) W) = (A f(H)) W: where the next layer is so much narrower that the
  // gathered bytes it saves outweigh a sweep for f(H), the product comes first and its few columns are propagated.  A gather
  // moves its entries at two to three times the sweep's rate; the line leaves that margin (13.8 k rows of 31 entries, 1000 to
  // 10 columns: objective 275 -> 152 us; 2.45 M rows of 51, 256 to 47: 25 -> 19 ms).  Else activations are taken as the rows are gathered.
  const float* forward_logits() {
    const float* h = H[1];
    if (!fresh) {
      gemm_nn(P[1], ld[0], P_max[1], W[1], ld[1], Wt[1], ld[0], B0, ld[1], n, C[1], C[0], img_H[1]);
      h = B0;
    }
    for (int l = 1; l < L; ++l) {
      float *const out = h == B0 ? B1 : B0, *const mid = out == B0 ? B1 : B0;
      float* const max = img_H[l + 1].data != nullptr ? B2_max : nullptr;
      if (gi.nnz * (long long)(ld[l] - ld[l + 1]) >= 8 * n * ld[l]) {
        relu(h, B2, ld[l], max);
        gemm_nn(B2, ld[l], max, W[l + 1], ld[l + 1], Wt[l + 1], ld[l], mid, ld[l + 1], n, C[l + 1], C[l], img_H[l + 1]);
        spmm(mid, out, ld[l + 1], nullptr);
      } else {
        spmm(h, B2, ld[l], max, true);
        gemm_nn(B2, ld[l], max, W[l + 1], ld[l + 1], Wt[l + 1], ld[l], out, ld[l + 1], n, C[l + 1], C[l], img_H[l + 1]);
      }
      h = out;
    }
    return h;
  }

  // Reported numbers and error flags, read back together.
  gk::Report read_report() {
    gk::Report r;
    CU(stage.get(&r, report, sizeof r, sizeof r, 1, stream));
    return r;
  }
  void check(const gk::Report& r) {
    if (r.error != 0) {   // a launch gave up and others may have left early: counters and products from scratch
      CU(cudaMemsetAsync(&report->error, 0, sizeof(int), stream));
      CU(cudaMemsetAsync(&report->status, 0, sizeof(int), stream));   // decisions since then may have read anything
      for (const auto& c : counters) CU(cudaMemsetAsync(*c.first, 0, c.second, stream));
      fresh = false;
      throw Fail{GCN_ADMM_ERR_CUDA, r.error & gk::kErrGridBarrier ? "a step-size search gave up waiting for the rest of its grid"
                                                                  : "a tensor-core product gave up waiting on its pipeline"};
    }
    if (r.status & 1) {
      CU(cudaMemsetAsync(&report->status, 0, sizeof(int), stream));
      throw Fail{GCN_ADMM_ERR_NONFINITE, "a non-finite value reached a step-size decision"};
    }
  }
  void check_status() { check(read_report()); }

  // rows in the caller's order (dense, width c) <-> internal (community order, padded).  Small matrices are written to and
  // read from the staging buffer by the permuting kernel itself.
  void rows_to_host(const float* dev, int c, float* host_out) {
    const size_t bytes = sizeof(float) * (size_t)n * c;
    const bool small = bytes <= kDirectBytes;
    char* near_host = nullptr;
    if (small) CU(stage.enter(stream, &near_host));
    float* dense = small ? reinterpret_cast<float*>(near_host) : B2;
    {
      Scope sc(this, "permute_rows", 1, 8.0 * (double)n * c, 0.0);
      gk::k_permute_rows<<<grid_for(n * ldpad(c)), 256, 0, stream>>>(dev, dense, d_inv, n, c, ldpad(c), 0);
      CU(cudaGetLastError());
    }
    if (small) {
      CU(stage.leave(stream));
      CU(cudaStreamSynchronize(stream));
      std::memcpy(host_out, near_host, bytes);
    } else {
      CU(stage.get(host_out, dense, bytes, bytes, 1, stream));
    }
  }
  void rows_from_host(const float* host_in, int c, float* dev) {
    const size_t bytes = sizeof(float) * (size_t)n * c;
    const bool small = bytes <= kDirectBytes;
    char* near_host = nullptr;
    const float* dense = B2;
    if (small) {
      CU(stage.enter(stream, &near_host));
      std::memcpy(near_host, host_in, bytes);
      dense = reinterpret_cast<const float*>(near_host);
    } else {
      CU(stage.put(B2, host_in, bytes, stream));
      CU(stage.flush(stream));
    }
    {
      Scope sc(this, "permute_rows", 1, 8.0 * (double)n * c, 0.0);
      gk::k_permute_rows<<<grid_for(n * ldpad(c)), 256, 0, stream>>>(dense, dev, d_inv, n, c, ldpad(c), 1);
      CU(cudaGetLastError());
    }
    if (small) CU(stage.leave(stream));
    else CU(stage.finish(stream));
  }
  // W_l and its transpose from a dense host matrix, through the gradient's buffer.
  void upload_weight(int l, const float* host_w) {
    const int r = C[l - 1], c = C[l];
    CU(stage.put(grad, host_w, sizeof(float) * (size_t)r * c, stream));
    CU(stage.finish(stream));
    const long long cells = std::max((long long)r * ld[l], (long long)c * ld[l - 1]);
    gk::WeightRange* const ranges = reinterpret_cast<gk::WeightRange*>(red_part);
    int n_ranges = 0;
    if (img_H[l].data != nullptr || img_G[l].data != nullptr) {
      n_ranges = (int)std::min<long long>(kSmCount, cdiv((long long)r * c, 256));
      gk::k_weight_range<<<n_ranges, 256, 0, stream>>>(grad, (long long)r * c, ranges);
    }
    gk::k_load_weight<<<grid_for(cells), 256, 0, stream>>>(grad, r, c, W[l], ld[l], Wt[l], ld[l - 1], img_H[l], img_G[l], ranges, n_ranges);
    CU(cudaGetLastError());
  }
  // Step parameters (t_prev) of `count` searches in a row, to and from the host.
  void take_steps(const SearchCtl* ctl, double* values, int count) {
    for (int k = 0; k < count; k += (int)(gcn_admm_mem::kSlot / sizeof(double))) {
      const int now = std::min(count - k, (int)(gcn_admm_mem::kSlot / sizeof(double)));
      char* near_host = nullptr;
      CU(stage.enter(stream, &near_host));
      gk::k_take_steps<<<(unsigned)cdiv(now, 256), 256, 0, stream>>>(ctl + k, reinterpret_cast<double*>(near_host), now);
      CU(cudaGetLastError());
      CU(stage.leave(stream));
      CU(cudaStreamSynchronize(stream));
      std::memcpy(values + k, near_host, sizeof(double) * now);
    }
  }
  void put_steps(SearchCtl* ctl, const double* values, int count) {
    for (int k = 0; k < count; k += (int)(gcn_admm_mem::kSlot / sizeof(double))) {
      const int now = std::min(count - k, (int)(gcn_admm_mem::kSlot / sizeof(double)));
      char* near_host = nullptr;
      CU(stage.enter(stream, &near_host));
      std::memcpy(near_host, values + k, sizeof(double) * now);
      gk::k_put_steps<<<(unsigned)cdiv(now, 256), 256, 0, stream>>>(ctl + k, reinterpret_cast<const double*>(near_host), now);
      CU(cudaGetLastError());
      CU(stage.leave(stream));
    }
  }
};

namespace {

template <typename F>
int guarded(gcn_admm* h, F&& body) {
  if (h == nullptr) return GCN_ADMM_ERR_ARG;
  try {
    cudaError_t e = cudaSetDevice(h->p.device);
    if (e != cudaSuccess) throw Fail{GCN_ADMM_ERR_CUDA, std::string("cudaSetDevice: ") + cudaGetErrorString(e)};
    body();
    return GCN_ADMM_OK;
  } catch (const Fail& f) {
    cudaGetLastError();   // reported here: the next call of this thread, on whichever handle, is not to find it again
    h->err = f.msg;
    return f.code;
  } catch (const std::bad_alloc&) {
    h->err = "host allocation failed";
    return GCN_ADMM_ERR_ALLOC;
  } catch (...) {
    h->err = "unexpected failure";
    return GCN_ADMM_ERR_CUDA;
  }
}

// View of `count` elements on the host: the caller's buffer itself when it is host memory, a copy when
// it lives on the device.
template <typename T>
struct HostView {
  gcn_admm_host::Table<T> copy;
  const T* ptr = nullptr;
  HostView(gcn_admm* h, const T* p, size_t count) {
    if (count > 0 && is_device_pointer(p)) {
      copy.resize(count);
      CU(cudaSetDevice(h->p.device));
      CU(cudaDeviceSynchronize());   // whatever fills the buffer, on whichever stream
      CU(h->stage.open());
      CU(h->stage.get(copy.data(), p, count * sizeof(T), count * sizeof(T), 1, h->stream));
      ptr = copy.data();
    } else {
      ptr = p;
    }
  }
  const T* data() const { return ptr; }
  const T& operator[](size_t i) const { return ptr[i]; }
};

void create_impl(gcn_admm* h, long long n, const long long* row_ptr, const int* col_idx, const float* X, const int* y,
                 const unsigned char* train_mask, int n_layers, const int* widths, int n_comm, const int* community) {
  const gcn_admm_params& p = h->p;
  h->L = n_layers;
  h->n = n;
  h->M = n_comm;
  h->C.assign(widths, widths + n_layers + 1);
  h->ld.resize(n_layers + 1);
  for (int l = 0; l <= n_layers; ++l) {
    if (h->C[l] < 1) throw Fail{GCN_ADMM_ERR_WIDTHS, "a layer width is smaller than 1"};
    h->ld[l] = ldpad(h->C[l]);
    h->max_ld = std::max(h->max_ld, h->ld[l]);
  }
  if (h->C[n_layers] > 32 * gk::kMaxClassesPerLane)
    throw Fail{GCN_ADMM_ERR_WIDTHS, "more than 128 classes are not supported"};
  for (int l = 2; l <= n_layers; ++l)
    if (h->ld[l] / 4 > 256) throw Fail{GCN_ADMM_ERR_WIDTHS, "layer widths above 1024 are supported for C_0 and C_1 only"};
  for (int l = 1; l <= n_layers; ++l)   // the Z scoring addresses rows of an N x C_l matrix by 32-bit float4 offsets
    if (n * (long long)(h->ld[l] / 4) >= (1LL << 32))
      throw Fail{GCN_ADMM_ERR_WIDTHS, "n x layer width exceeds 2^34 elements"};

  // host copies of the graph-side inputs, then the index tables
  h->stream = static_cast<cudaStream_t>(p.stream);
  HostView<long long> rp(h, row_ptr, (size_t)n + 1);
  if (rp[n] < 0 || rp[0] != 0) throw Fail{GCN_ADMM_ERR_GRAPH, "row_ptr must start at 0 and be ascending"};
  HostView<int> ci(h, col_idx, (size_t)rp[n]);
  HostView<int> comm(h, community, (size_t)n);
  HostView<int> yy(h, y, (size_t)n);
  HostView<unsigned char> tm(h, train_mask, (size_t)n);
  std::string msg;
  const int rc = gcn_admm_host::build_graph_index(n, rp.data(), ci.data(), n_comm, comm.data(), h->gi, msg);
  if (rc == gcn_admm_host::IDX_BAD_GRAPH) throw Fail{GCN_ADMM_ERR_GRAPH, msg};
  if (rc == gcn_admm_host::IDX_BAD_COMMUNITY) throw Fail{GCN_ADMM_ERR_COMMUNITY, msg};
  { gcn_admm_host::Table<long long>().swap(rp.copy); gcn_admm_host::Table<int>().swap(ci.copy); }
  const GraphIndex& g = h->gi;
  gcn_admm_host::Table<int> y_new;
  gcn_admm_host::Table<unsigned char> t_new;
  y_new.resize((size_t)n);
  t_new.resize((size_t)n);
  int bad_label = 0, n_train = 0;
#pragma omp parallel for schedule(static) reduction(| : bad_label) reduction(+ : n_train) if (n > 20000)
  for (long long i = 0; i < n; ++i) {
    const bool in = yy[g.perm[i]] >= 0 && yy[g.perm[i]] < h->C[n_layers];
    t_new[(size_t)i] = tm[g.perm[i]] ? 1 : 0;
    n_train += t_new[(size_t)i];
    bad_label |= t_new[(size_t)i] && !in;
    y_new[(size_t)i] = in ? yy[g.perm[i]] : 0;
  }
  h->n_train = n_train;
  if (bad_label) throw Fail{GCN_ADMM_ERR_WIDTHS, "a training label lies outside 0..C_L-1"};
  // all host-side validation is done; from here on a CUDA device is required
  int dev_count = 0;
  CU(cudaGetDeviceCount(&dev_count));
  if (p.device < 0 || p.device >= dev_count) throw Fail{GCN_ADMM_ERR_CUDA, "no such CUDA device"};
  CU(cudaSetDevice(p.device));
  CU(h->stage.open());
  h->want_table(h->d_row_ptr, g.row_ptr);
  h->want_table(h->d_col, g.col);
  h->want_table(h->d_row_comm, g.row_comm);
  h->want_table(h->d_perm, g.perm);
  h->want_table(h->d_inv, g.inv);
  h->want_table(h->d_dinv, g.dinv);
  h->want_table(h->d_col_comm, g.col_comm);
  h->want_table(h->d_y, y_new);
  h->want_table(h->d_train, t_new);
  std::vector<int> tr;
  tr.reserve((size_t)h->n_train);
  for (long long i = 0; i < n; ++i)
    if (t_new[(size_t)i]) tr.push_back((int)i);
  h->want_table(h->d_train_rows, tr);
  std::vector<float> mom((size_t)std::max(p.fista_iters, 1), 0.f);
  {
    double t = 1.0;
    for (int j = 0; j < p.fista_iters; ++j) {
      const double tn = 0.5 * (1.0 + std::sqrt(1.0 + 4.0 * t * t));
      mom[(size_t)j] = (float)((t - 1.0) / tn);
      t = tn;
    }
  }
  h->want_table(h->d_fista_momentum, mom);
  h->long_len = p.long_row > 0 ? p.long_row : default_long_row(n, g.nnz);
  gcn_admm_host::LongRowTables lt;
  gcn_admm_host::build_long_row_tables(g, h->long_len, lt);
  h->n_items = (int)lt.items.size();
  h->n_split = (int)lt.split.size();
  h->n_long = (int)lt.rows.size();
  h->want_table(h->d_items, lt.items);
  h->want_table(h->d_split, lt.split);
  h->want_table(h->d_long_rows, lt.rows);
  std::vector<int> item_row(lt.items.size());
  for (size_t r = 0; r < lt.rows.size(); ++r)
    for (int k = 0; k < lt.rows[r].z; ++k) item_row[(size_t)(lt.rows[r].y + k)] = (int)r;
  h->want_table(h->d_item_row, item_row);
  h->want_counter(h->d_row_done, lt.rows.size());
  // split entries grouped by community (stable), for the ordered sums of the Z search
  std::vector<int> split_ptr((size_t)n_comm + 1, 0), split_order(lt.split.size());
  for (const auto& q : lt.split) ++split_ptr[(size_t)q.y + 1];
  for (int m = 0; m < n_comm; ++m) split_ptr[m + 1] += split_ptr[m];
  {
    std::vector<int> at(split_ptr.begin(), split_ptr.end() - 1);
    for (size_t k = 0; k < lt.split.size(); ++k) split_order[(size_t)at[lt.split[k].y]++] = (int)k;
  }
  h->want_table(h->d_split_order, split_order);
  h->want_table(h->d_split_ptr, split_ptr);
  h->want(h->split_scores, lt.split.size() * gk::kCand);
  gcn_admm_host::Table<int> row_order;
  gcn_admm_host::order_rows_by_length(g, row_order);
  h->want_table(h->d_row_order, row_order);
  h->want(h->d_row_table, (size_t)n);
  if ((long long)g.nnz <= kUserColumns) h->want(h->d_user_col, (size_t)g.nnz);
  // work lists of the two forms of the Z search: the closed form's segments by community (at least two layers), and chunks
  // of units (items first, then rows) holding about the same number of stored entries each (at least three layers)
  gcn_admm_host::SegmentTables seg;
  std::vector<int> chunks;
  const long long warps_guess = (long long)kSmCount * 3 * 8;
  if (n_layers >= 2) {
    // a chunk per warp and a few more; rows of the plain sums in chunks of about 8 KB
    const long long target = std::max<long long>(32, std::min<long long>(1024, (long long)g.nnz / (warps_guess * 2)));
    gcn_admm_host::build_segment_tables(g, h->long_len, lt, target, std::max(1, 2048 / h->ld[n_layers]), seg);
    static_assert(sizeof(gcn_admm_host::SegRef) == sizeof(gk::SegRef) && sizeof(gcn_admm_host::SegChunk) == sizeof(gk::SegChunk),
                  "tables are uploaded as they are");
    h->n_seg_chunks = (int)seg.chunks.size();
    h->want_table(h->d_segs, seg.segs);
    h->want_table(h->d_seg_chunks, seg.chunks);
    h->want_table(h->d_slot_ptr, seg.slot_ptr);
    h->want(h->slots, 2 * (size_t)seg.slot_ptr.back());
    h->want_counter(h->comm_done, n_comm);
    h->want_counter(h->split_done, lt.split.size());
  }
  if (n_layers >= 3) {
    const long long n_units = (long long)lt.items.size() + n;
    // few enough chunks that their sums (M x candidates doubles each) stay small next to the entries they cover
    const long long target = std::max<long long>({64, std::min<long long>(1024, (long long)g.nnz / (warps_guess * 4)), 2LL * n_comm});
    chunks.push_back(0);
    long long in_chunk = 0;
    for (long long u = 0; u < n_units; ++u) {
      long long len;
      if (u < (long long)lt.items.size()) len = lt.items[(size_t)u].z - lt.items[(size_t)u].y;
      else {
        const long long r = u - (long long)lt.items.size();
        len = g.row_ptr[r + 1] - g.row_ptr[r];
        if (len > h->long_len) len = 0;                 // walked as items
      }
      in_chunk += len + 2;                              // a unit costs a little even when it is short
      if (in_chunk >= target) { chunks.push_back((int)(u + 1)); in_chunk = 0; }
    }
    if (chunks.back() != (int)n_units) chunks.push_back((int)n_units);
  }
  h->n_chunks = std::max(0, (int)chunks.size() - 1);
  h->want_table(h->d_chunk_ptr, chunks);

  const int L = n_layers;
  const size_t rows = (size_t)n;
  h->W.assign(L + 1, nullptr); h->Wt.assign(L + 1, nullptr); h->Z.assign(L + 1, nullptr);
  h->P.assign(L + 1, nullptr); h->H.assign(L + 1, nullptr);
  size_t grad_elems = 1, grad_t_elems = 1, grad_blocks = 1;   // grad_blocks: most blocks of a finish_grad launch
  h->part_elems = 1;
  for (int l = 1; l <= L; ++l) {
    h->want(h->W[l], (size_t)h->C[l - 1] * h->ld[l]);
    h->want(h->Wt[l], (size_t)h->C[l] * h->ld[l - 1]);
    h->want(h->Z[l], rows * h->ld[l]);
    h->want(h->P[l], rows * h->ld[l - 1]);
    h->want(h->H[l], rows * h->ld[l]);
    const size_t ge = (size_t)h->C[l - 1] * h->ld[l];
    grad_elems = std::max(grad_elems, ge);
    grad_blocks = std::max(grad_blocks, (size_t)cdiv((long long)ge, 32));
    grad_t_elems = std::max(grad_t_elems, (size_t)h->C[l] * h->ld[l - 1]);
    h->part_elems = std::max(h->part_elems, ge * 4 * kSmCount);
  }
  for (int l = 1; l <= L; ++l)   // room for one split per 2048 rows (tensor-core form of the transposed product)
    h->part_elems = std::max(h->part_elems, (size_t)h->C[l - 1] * h->ld[l] * (size_t)(cdiv(n, 2048) + kSmCount));
  h->part_elems = std::min<size_t>(h->part_elems, (size_t)256 << 20);   // at most 1 GB of partial sums
  h->part_elems = std::max(h->part_elems, grad_elems);
  h->want(h->U, rows * h->ld[L], gcn_admm::kZero);
  h->want(h->B0, rows * h->max_ld);
  h->want(h->B1, rows * h->max_ld);
  h->want(h->B2, rows * h->max_ld);
  // a second line of launches where a pass is short enough for it to matter (the sizes that are recorded as graphs)
  h->two_lanes = L >= 2 && n * (long long)h->max_ld < kSmallProblem;
  if (h->two_lanes) {
    const size_t ge = (size_t)h->C[L - 1] * h->ld[L];
    h->want(h->RL, rows * h->ld[L]);
    h->want(h->DL, rows * h->ld[L]);
    h->side.part_elems = std::max<size_t>(ge, std::min<size_t>(std::max(ge * 4 * kSmCount, ge * (size_t)(cdiv(n, 2048) + kSmCount)), (size_t)64 << 20));
    h->want(h->side.part, h->side.part_elems);
    h->want(h->side.grad, ge);
    h->want(h->side.grad_t, (size_t)h->C[L] * h->ld[L - 1], gcn_admm::kZero);
    h->want(h->side.red_part, std::max<size_t>((size_t)kSmCount * 8 * gk::kCand, (size_t)cdiv((long long)ge, 32) * 3));
    h->want_counter(h->side.ticket, 1);
    h->want_counter(h->side.tile_tickets, kSmCount);
    CU(gcn_admm_mem::Pool::get().take_stream(p.device, &h->side.stream));
    for (cudaEvent_t* e : {&h->side.begun, &h->side.w_done, &h->side.out_done, &h->side.done}) CU(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  }
  h->item_sums_elems = std::max<size_t>(1, (size_t)h->n_items * h->max_ld);
  h->want(h->item_sums, h->item_sums_elems);
  h->want(h->grad, grad_elems);
  h->want(h->grad_t, grad_t_elems, gcn_admm::kZero);
  h->img_H.assign(L + 1, gtc::Image{nullptr, 16, 1}); h->img_G = h->img_D = h->img_H;
  h->P_max.assign(L + 1, nullptr);
  for (int l = 1; l <= L; ++l) {
    h->want_image(h->img_H[l], h->C[l], h->C[l - 1]);   // P_l W_l, G W_l; P_l grad has its shape
    h->want_image(h->img_D[l], h->C[l], h->C[l - 1]);
    if (l >= 2 && !h->joins_products(l - 1)) h->want_image(h->img_G[l], h->C[l - 1], h->C[l]);   // (narrower: k_zgrad_products)
    if (h->by_halves(n, h->C[l], h->C[l - 1])) h->want(h->P_max[l], rows);
  }
  h->want(h->B1_max, rows);
  h->want(h->B2_max, rows);
  h->want(h->part, h->part_elems);
  std::vector<SearchCtl> cw(L + 1), cz((size_t)(L + 1) * n_comm);
  std::memset(cw.data(), 0, cw.size() * sizeof(SearchCtl));
  std::memset(cz.data(), 0, cz.size() * sizeof(SearchCtl));
  for (auto& c : cw) { c.t_prev = p.tau0; c.done = 1; c.trial = -3; }
  for (auto& c : cz) { c.t_prev = p.theta0; c.done = 1; c.trial = -3; }
  h->want_table(h->ctl_w, cw);
  h->want_table(h->ctl_z, cz);
  h->want(h->sums_z, (size_t)3 * n_comm);
  h->want(h->report, 1, gcn_admm::kZero);
  // row blocks of the hidden-layer gradient's closing sweep, cut at community boundaries
  std::vector<int4> zb;
  std::vector<int> cbp((size_t)n_comm + 1, 0);
  for (int m = 0; m < n_comm; ++m) {
    cbp[m] = (int)zb.size();
    for (int r = g.comm_ptr[m]; r < g.comm_ptr[m + 1]; r += kZBlockRows)
      zb.push_back(make_int4(r, std::min(r + kZBlockRows, g.comm_ptr[m + 1]), m, 0));
  }
  cbp[n_comm] = (int)zb.size();
  h->n_zblocks = (int)zb.size();
  h->want_table(h->d_zblocks, zb);
  h->want_table(h->d_comm_block_ptr, cbp);
  h->want(h->z_chunk_part, (size_t)h->n_chunks * n_comm * gk::kCand);
  h->want(h->z_group_part, (size_t)kChunkGroups * n_comm * gk::kCand);
  h->want_counter(h->chunk_counter, 1);
  h->want_counter(h->ticket, 1);
  h->want_counter(h->tile_tickets, kSmCount);
  h->want_counter(h->comm_tickets, n_comm);
  h->want_counter(h->grid_bar, 1);
  h->want(h->red_part, std::max<size_t>({(size_t)kSmCount * 8 * gk::kCand, (size_t)h->n_zblocks * 3,
                                         (size_t)cdiv(n, 8) * 2, grad_blocks * 3}));
  h->want_counter(h->n_active, 1);
  h->want(h->d_pass, 1, gcn_admm::kZero);
  h->want(h->d_h1_age, 1, gcn_admm::kZero);
  h->want(h->skip_h1, 1, gcn_admm::kZero);
  h->want(h->log_trial_w, (size_t)kLogPasses * L);
  h->want(h->log_q_w, (size_t)kLogPasses * L);
  h->want(h->log_trial_z, (size_t)kLogPasses * std::max(L - 1, 0) * n_comm);
  h->want(h->log_q_z, (size_t)kLogPasses * std::max(L - 1, 0) * n_comm);
  h->commit();
  { gcn_admm_host::Table<unsigned short>().swap(h->gi.col_comm); }   // needed on the device only
  h->status = &h->report->status;
  h->tc_error = &h->report->error;
  {
    gcn_admm::Scope sc(h, "gather_tables", 1, 24.0 * n + 12.0 * g.nnz, 0.0);
    gk::k_gather_tables<<<h->grid_for(std::max<long long>(n, h->d_user_col ? g.nnz : 0)), 256, 0, h->stream>>>(
        h->d_row_order, h->d_row_ptr, h->d_dinv, (int)n, h->d_row_table, h->d_col, h->d_perm, g.nnz, h->d_user_col);
    CU(cudaGetLastError());
  }

  // Z_0 in community order, then P_1 = A~ Z_0 (Z_0 never changes, so neither does P_1)
  {
    const bool on_device = is_device_pointer(X);
    if (on_device) CU(cudaDeviceSynchronize());
    else CU(h->stage.put(h->B0, X, rows * h->C[0] * sizeof(float), h->stream));
    CU(h->stage.flush(h->stream));
    {
      gcn_admm::Scope sc(h, "permute_rows", 1, 8.0 * (double)n * h->C[0], 0.0);
      gk::k_permute_rows<<<h->grid_for(n * h->ld[0]), 256, 0, h->stream>>>(on_device ? X : h->B0, h->B1, h->d_inv, n, h->C[0], h->ld[0], 1);
      CU(cudaGetLastError());
    }
    h->spmm(h->B1, h->P[1], h->ld[0], h->P_max[1]);
  }

  for (int l = 1; l <= L; ++l) {
    if (p.w_init != nullptr) { h->upload_weight(l, p.w_init[l - 1]); continue; }
    // no weights given: Glorot-uniform from a counter-based generator (see the header for the definition)
    const int r = h->C[l - 1], c = h->C[l];
    std::vector<float> w((size_t)r * c);
    const double a = std::sqrt(6.0 / ((double)r + (double)c));
    for (size_t e = 0; e < w.size(); ++e) {
      const double u = (double)(splitmix64(p.seed + ((unsigned long long)l << 32) + e) >> 40) / 16777216.0;
      w[e] = (float)(a * (2.0 * u - 1.0));
    }
    h->upload_weight(l, w.data());
  }
  // forward pass of Problem 1 with the same kernels that later recompute H_l, so that the
  // initial residuals are exactly zero
  for (int l = 1; l <= L; ++l) {
    if (l >= 2) h->spmm(h->Z[l - 1], h->P[l], h->ld[l - 1], h->P_max[l]);
    h->refresh_H(l);
    if (l < L) h->relu(h->H[l], h->Z[l], h->ld[l]);
    else CU(cudaMemcpyAsync(h->Z[l], h->H[l], rows * h->ld[l] * sizeof(float), cudaMemcpyDeviceToDevice, h->stream));
  }
  h->fresh = true;
  CU(h->stage.finish(h->stream));
  CU(cudaStreamSynchronize(h->stream));
}

}  // namespace

extern "C" {

void gcn_admm_default_params(gcn_admm_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->nu = 1e-3f; p->rho = 1e-3f;
  p->tau0 = 1.f; p->theta0 = 1.f;
  p->bt_growth = 2.f; p->bt_shrink = 0.5f;
  p->bt_max_trials = 40;
  p->fista_iters = 30;
  p->loss_scale = 1.f;
  p->dual_mode = 0;
  p->tensor_cores = 1;
  p->use_graph = 2;
  p->schedule = 0;
  p->long_row = 0;
  p->seed = 0;
  p->w_init = nullptr;
  p->device = 0;
  p->stream = nullptr;
}

int gcn_admm_create(gcn_admm** out, long long n, const long long* row_ptr, const int* col_idx, const float* X,
                    const int* y, const unsigned char* train_mask, int n_layers, const int* widths,
                    const gcn_admm_params* p, int n_comm, const int* community) {
  if (out) *out = nullptr;
  if (!out || !row_ptr || !X || !y || !train_mask || !widths || !p || !community || !col_idx) {
    g_create_error = "NULL argument";
    return GCN_ADMM_ERR_ARG;
  }
  if (n < 1 || n > 2147483647LL / 2 || n_comm < 1) { g_create_error = "n and n_comm must be positive"; return GCN_ADMM_ERR_ARG; }
  if (n_comm > 65535) { g_create_error = "more than 65535 communities are not supported"; return GCN_ADMM_ERR_COMMUNITY; }
  if (n_layers < 1 || n_layers > 64) { g_create_error = "n_layers must be 1..64"; return GCN_ADMM_ERR_WIDTHS; }
  for (int l = 0; p->w_init && l < n_layers; ++l)
    if (!p->w_init[l]) { g_create_error = "w_init holds a NULL pointer"; return GCN_ADMM_ERR_ARG; }
  if (!(p->nu > 0.f) || !(p->rho > 0.f) || !(p->bt_growth > 1.f) || !(p->bt_shrink > 0.f) || p->bt_max_trials < 1 ||
      p->bt_max_trials > 64 || p->fista_iters < 0 || p->schedule < 0 || p->schedule > 1 || p->long_row < 0 || !(p->tau0 > 0.f) || !(p->theta0 > 0.f) || !(p->loss_scale > 0.f)) {
    g_create_error = "a parameter is out of range";
    return GCN_ADMM_ERR_ARG;
  }
  gcn_admm* h = new (std::nothrow) gcn_admm();
  if (!h) { g_create_error = "host allocation failed"; return GCN_ADMM_ERR_ALLOC; }
  h->p = *p;
  int code = GCN_ADMM_OK;
  try {
    create_impl(h, n, row_ptr, col_idx, X, y, train_mask, n_layers, widths, n_comm, community);
  } catch (const Fail& f) {
    code = f.code; g_create_error = f.msg;
  } catch (const std::bad_alloc&) {
    code = GCN_ADMM_ERR_ALLOC; g_create_error = "host allocation failed";
  } catch (...) {
    code = GCN_ADMM_ERR_CUDA; g_create_error = "unexpected failure";
  }
  if (code != GCN_ADMM_OK) {
    gcn_admm_destroy(h);
    return code;
  }
  h->p.w_init = nullptr;   // the caller's pointers are not kept
  *out = h;
  return GCN_ADMM_OK;
}

void gcn_admm_destroy(gcn_admm* h) {
  if (!h) return;
  if (cudaSetDevice(h->p.device) == cudaSuccess) {
    cudaStreamSynchronize(h->stream);
    for (const ProfPending& q : h->pending)
      for (cudaEvent_t e : {q.a, q.b}) cudaEventDestroy(e);
    if (h->pass_graph) cudaGraphExecDestroy(h->pass_graph);
    if (h->side.stream) {
      cudaStreamSynchronize(h->side.stream);
      gcn_admm_mem::Pool::get().give_stream(h->p.device, h->side.stream);
    }
    for (cudaEvent_t e : {h->side.begun, h->side.w_done, h->side.out_done, h->side.done})
      if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : h->event_pool) cudaEventDestroy(e);
    for (const gcn_admm_mem::Slab& q : {h->slab, h->wide_sums}) gcn_admm_mem::Pool::get().give(q);
    h->stage.close();
  }
  cudaGetLastError();
  delete h;
}

void gcn_admm_release_idle(void) {
  gcn_admm_mem::Pool::get().release();
  cudaGetLastError();
}

const char* gcn_admm_last_error(const gcn_admm* h) { return h ? h->err.c_str() : g_create_error.c_str(); }

int gcn_admm_step(gcn_admm* h, int n_iters) {
  return guarded(h, [&] {
    if (n_iters < 0) throw Fail{GCN_ADMM_ERR_ARG, "n_iters must be >= 0"};
    h->log_count = 0;
    CU(cudaMemsetAsync(h->d_pass, 0, sizeof(int), h->stream));
    // A pass is a fixed sequence of launches (every decision is taken on the device), so on a stream
    // that can be captured it is recorded once and replayed: the small workloads are launch-bound.
    // use_graph 1: always; 2: only where a pass is short enough for launch overhead to matter
    const bool wanted = h->p.use_graph == 1 || (h->p.use_graph == 2 && h->n * (long long)h->max_ld < kSmallProblem);
    // single passes are recorded once a few of them have been asked for: a loop that looks at the result after each
    const bool replay = wanted && h->stream != nullptr && !h->profiling && n_iters >= 1 &&
                        (n_iters >= 2 || h->pass_graph != nullptr || h->single_passes >= 2);
    if (!replay) {
      for (int k = 0; k < n_iters; ++k) h->iterate();
      h->single_passes += n_iters;
      return;
    }
    if (!h->fresh) h->refresh();
    if (h->pass_graph == nullptr) {
      cudaGraph_t graph = nullptr;
      CU(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
      const long long launches_before = h->launches, log_before = h->log_count;
      h->capturing = true;          // it launches every product; the device leaves H_1's out while H_1 is kept (see refresh)
      try {
        h->iterate();
        h->capturing = false;
      } catch (...) {
        h->capturing = false;
        cudaStreamEndCapture(h->stream, &graph);
        if (graph) cudaGraphDestroy(graph);
        throw;
      }
      CU(cudaStreamEndCapture(h->stream, &graph));
      h->launches_per_pass = h->launches - launches_before;
      h->launches = launches_before;       // recording launched nothing
      h->log_count = log_before;
      cudaError_t e = cudaGraphInstantiate(&h->pass_graph, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) throw Fail{GCN_ADMM_ERR_CUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e)};
    }
    for (int k = 0; k < n_iters; ++k) {
      CU(cudaGraphLaunch(h->pass_graph, h->stream));
      h->launches += h->launches_per_pass;
      ++h->log_count;
    }
  });
}

int gcn_admm_step_block(gcn_admm* h, int phase, int layer) {
  return guarded(h, [&] {
    const int L = h->L;
    if (phase == GCN_ADMM_PHASE_W || phase == GCN_ADMM_PHASE_Z)
      if (layer < 1 || layer > L) throw Fail{GCN_ADMM_ERR_ARG, "layer out of range"};
    if (!h->fresh) h->refresh();
    h->log_count = 0;
    CU(cudaMemsetAsync(h->d_pass, 0, sizeof(int), h->stream));
    h->clear_log_pass();
    if (phase == GCN_ADMM_PHASE_W) {
      h->update_W(layer, false);
    } else if (phase == GCN_ADMM_PHASE_Z) {
      if (layer < L) h->update_Z_hidden(layer, false);
      else h->update_output(false, true);
      h->fresh = false;
    } else if (phase == GCN_ADMM_PHASE_U) {
      h->dual_from_stored();
    } else {
      throw Fail{GCN_ADMM_ERR_ARG, "unknown phase"};
    }
    h->log_count = 1;
  });
}

int gcn_admm_objective(gcn_admm* h, double out[6]) {
  return guarded(h, [&] {
    if (!out) throw Fail{GCN_ADMM_ERR_ARG, "NULL output"};
    if (!h->fresh) h->refresh();
    const int L = h->L;
    double* const obj = h->report->obj;
    for (int l = 1; l < L; ++l) {
      const long long n4 = h->n * h->ld[l] / 4;
      gcn_admm::Scope sc(h, "objective_sums", 1, 32.0 * n4, 0.0);
      h->launch(gk::k_sum_hidden_penalty, h->grid_for(n4), 256, 0, (const float4*)h->Z[l], (const float4*)h->H[l], n4, h->red_part, h->ticket, obj + 2, l > 1);
    }
    const long long n4 = h->n * h->ld[L] / 4;
    const int row_blocks = h->grid_for(8 * h->n);   // eight lanes per row
    {
      gcn_admm::Scope sc_obj(h, "objective_sums", 2, 48.0 * n4, 0.0);
      h->launch(gk::k_sum_constraint, h->grid_for(n4), 256, 0, (const float4*)h->Z[L], (const float4*)h->H[L], (const float4*)h->U, n4, h->red_part,
                h->ticket, obj + 3);
      h->launch(gk::k_row_loss_argmax, row_blocks, 256, 0, (const float4*)h->Z[L], nullptr, h->ld[L] / 4, h->C[L], (int)h->n, h->d_y, h->d_train, nullptr,
                nullptr, h->red_part, h->ticket, obj);            // obj[0] = cross-entropy sum
      CU(cudaGetLastError());
    }
    const float* const logits = h->forward_logits();
    {
      gcn_admm::Scope sc_obj(h, "objective_sums", 1, 4.0 * (double)h->n * h->ld[L], 0.0);
      h->launch(gk::k_row_loss_argmax, row_blocks, 256, 0, nullptr, (const float4*)logits, h->ld[L] / 4, h->C[L], (int)h->n, h->d_y, h->d_train, nullptr,
                nullptr, h->red_part, h->ticket, obj + 5);        // obj[6] = correct training rows
      CU(cudaGetLastError());
    }
    const gk::Report report = h->read_report();
    const double* const v = report.obj;
    const double R = h->p.loss_scale * v[0];
    const double pen = L > 1 ? 0.5 * h->p.nu * v[2] : 0.0;
    const double ur = v[3];
    const double rr = 0.5 * h->p.rho * v[4];
    out[0] = R + pen + ur + rr;
    out[1] = R; out[2] = pen; out[3] = ur; out[4] = rr;
    out[5] = h->n_train > 0 ? v[6] / h->n_train : 0.0;
    h->check(report);
  });
}

int gcn_admm_weights(gcn_admm* h, int layer, float* out) {
  return gcn_admm_get_state(h, GCN_ADMM_ST_W, layer, out);
}

int gcn_admm_predict(gcn_admm* h, float* logits, int* labels) {
  return guarded(h, [&] {
    const int L = h->L, C = h->C[L];
    const size_t label_bytes = labels ? sizeof(int) * (size_t)h->n : 0, logit_bytes = logits ? sizeof(float) * (size_t)h->n * C : 0;
    const float* const z = h->forward_logits();
    // Labels and logits leave together: one wait where they are small (the kernels write page-locked memory), and else the bus takes
    // the logits while the host still empties the labels (one after the other 55 us of 1.3 ms at 169 k rows of 40 classes).
    const bool small = label_bytes + logit_bytes <= kDirectBytes;
    char* near_host = nullptr;
    if (small) CU(h->stage.enter(h->stream, &near_host));
    float* const dense = small ? reinterpret_cast<float*>(near_host) : h->B2;
    int* const d_lab = small ? reinterpret_cast<int*>(near_host + logit_bytes) : reinterpret_cast<int*>(z == h->B0 ? h->B1 : h->B0);
    if (labels) {
      gcn_admm::Scope sc(h, "row_argmax", 1, 4.0 * (double)h->n * h->ld[L], 0.0);
      h->launch(gk::k_row_loss_argmax, h->grid_for(8 * h->n), 256, 0, nullptr, (const float4*)z, h->ld[L] / 4, C, (int)h->n, h->d_y, h->d_train,
                d_lab, h->d_perm, nullptr, nullptr, nullptr);
      CU(cudaGetLastError());
    }
    if (logits) {
      gcn_admm::Scope sc(h, "permute_rows", 1, 8.0 * (double)h->n * C, 0.0);
      gk::k_permute_rows<<<h->grid_for(h->n * h->ld[L]), 256, 0, h->stream>>>(z, dense, h->d_inv, h->n, C, h->ld[L], 0);
      CU(cudaGetLastError());
    }
    if (small) {
      CU(h->stage.leave(h->stream));
      CU(cudaStreamSynchronize(h->stream));
      if (logits) std::memcpy(logits, dense, logit_bytes);
      if (labels) std::memcpy(labels, d_lab, label_bytes);
    } else {
      const gcn_admm_mem::Stage::Part parts[2] = {{labels, d_lab, label_bytes}, {logits, dense, logit_bytes}};
      CU(h->stage.get_all(parts, 2, h->stream));
    }
    CU(cudaStreamSynchronize(h->stream));
  });
}

int gcn_admm_propagate(gcn_admm* h, const float* x, int width, float* out) {
  return guarded(h, [&] {
    if (!x || !out || width < 1 || width > kMaxWidth) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    const bool dev_in = is_device_pointer(x), dev_out = is_device_pointer(out);
    if (dev_in != dev_out) throw Fail{GCN_ADMM_ERR_ARG, "x and out must both be host or both be device pointers"};
    h->grow_wide_sums(ldpad(width));
    if (dev_in) {
      h->propagate_dense(x, width, out, true);
      CU(cudaStreamSynchronize(h->stream));
      return;
    }
    // host buffers: staged in two of the handle's scratch matrices (idle between calls), or, wider than those, in
    // a pair allocated for the call
    const size_t elems = (size_t)h->n * width, bytes = elems * sizeof(float);
    const bool fits = width <= h->max_ld;
    float *a = fits ? h->B0 : dalloc<float>(elems), *b = nullptr;
    try {
      b = fits ? h->B1 : dalloc<float>(elems);
      CU(h->stage.put(a, x, bytes, h->stream));
      CU(h->stage.flush(h->stream));
      h->propagate_dense(a, width, b, true);
      CU(h->stage.get(out, b, bytes, bytes, 1, h->stream));
      CU(h->stage.finish(h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } catch (...) {
      if (!fits) { cudaFree(a); cudaFree(b); }
      throw;
    }
    if (!fits) { cudaFree(a); cudaFree(b); }
  });
}

int gcn_admm_dense_product(gcn_admm* h, const float* A, const float* B, float* C, long long m, int n, int k,
                           int tensor_cores) {
  return guarded(h, [&] {
    if (!A || !B || !C || m < 1 || n < 1 || k < 1 || m > 2147483647LL) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    if (!is_device_pointer(A) || !is_device_pointer(B) || !is_device_pointer(C))
      throw Fail{GCN_ADMM_ERR_ARG, "A, B and C must be device pointers"};
    const int lda = ldpad(k), ldb = ldpad(n), ldc = ldpad(n), ldbk = ldpad(k);
    float *a = nullptr, *b = nullptr, *bk = nullptr, *c = nullptr, *a_max = nullptr;
    gtc::Image image{nullptr, 16, 1};
    const int saved = h->p.tensor_cores;
    try {
      a = dalloc<float>((size_t)m * lda);
      b = dalloc<float>((size_t)k * ldb);
      bk = dalloc<float>((size_t)n * ldbk);
      c = dalloc<float>((size_t)m * ldc);
      CU(cudaMemsetAsync(a, 0, (size_t)m * lda * 4, h->stream));
      CU(cudaMemsetAsync(b, 0, (size_t)k * ldb * 4, h->stream));
      CU(cudaMemsetAsync(bk, 0, (size_t)n * ldbk * 4, h->stream));
      CU(cudaMemcpy2DAsync(a, (size_t)lda * 4, A, (size_t)k * 4, (size_t)k * 4, (size_t)m, cudaMemcpyDeviceToDevice, h->stream));
      CU(cudaMemcpy2DAsync(b, (size_t)ldb * 4, B, (size_t)n * 4, (size_t)n * 4, (size_t)k, cudaMemcpyDeviceToDevice, h->stream));
      gk::k_transpose_small<<<(unsigned)cdiv((long long)k * n, 256), 256, 0, h->stream>>>(b, ldb, bk, ldbk, k, n);
      CU(cudaGetLastError());
      h->p.tensor_cores = tensor_cores;
      if (tensor_cores && h->by_halves(m, n, k)) {
        image.nt = gcn_admm::group_width(n, true);
        image.kc = (int)cdiv(k, gtc::kChunkK);
        image.data = dalloc<uint8_t>(gcn_admm::image_bytes(n, image));
        CU(cudaMemsetAsync(image.data, 0, gcn_admm::image_bytes(n, image), h->stream));
        a_max = dalloc<float>((size_t)m);
        h->split_b(gtc::SplitB{bk, ldbk, n, k, image});
        gk::k_row_max<<<h->grid_for(32 * m), 256, 0, h->stream>>>(reinterpret_cast<const float4*>(a), lda / 4, m, a_max);
        CU(cudaGetLastError());
        ++h->launches;
      }
      h->gemm_nn(a, lda, a_max, b, ldb, tensor_cores ? bk : nullptr, ldbk, c, ldc, m, n, k, image);
      h->p.tensor_cores = saved;
      CU(cudaMemcpy2DAsync(C, (size_t)n * 4, c, (size_t)ldc * 4, (size_t)n * 4, (size_t)m, cudaMemcpyDeviceToDevice, h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } catch (...) {
      h->p.tensor_cores = saved;
      cudaFree(a); cudaFree(b); cudaFree(bk); cudaFree(c); cudaFree(a_max); cudaFree(image.data);
      throw;
    }
    cudaFree(a); cudaFree(b); cudaFree(bk); cudaFree(c); cudaFree(a_max); cudaFree(image.data);
    h->check_status();
  });
}

int gcn_admm_dense_product_tn(gcn_admm* h, const float* A, const float* B, float* C, long long rows, int ka, int nb,
                              int tensor_cores) {
  return guarded(h, [&] {
    if (!A || !B || !C || rows < 1 || ka < 1 || nb < 1) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    if (!is_device_pointer(A) || !is_device_pointer(B) || !is_device_pointer(C))
      throw Fail{GCN_ADMM_ERR_ARG, "A, B and C must be device pointers"};
    const int lda = ldpad(ka), ldb = ldpad(nb), ldp = ldpad(nb);
    if ((size_t)ka * ldp > h->part_elems) throw Fail{GCN_ADMM_ERR_ARG, "ka x nb exceeds the handle's partial-sum scratch"};
    float *a = nullptr, *b = nullptr, *c = nullptr;
    const int saved = h->p.tensor_cores;
    try {
      a = dalloc<float>((size_t)rows * lda);
      b = dalloc<float>((size_t)rows * ldb);
      c = dalloc<float>((size_t)ka * ldp);
      CU(cudaMemsetAsync(a, 0, (size_t)rows * lda * 4, h->stream));
      CU(cudaMemsetAsync(b, 0, (size_t)rows * ldb * 4, h->stream));
      CU(cudaMemcpy2DAsync(a, (size_t)lda * 4, A, (size_t)ka * 4, (size_t)ka * 4, (size_t)rows, cudaMemcpyDeviceToDevice, h->stream));
      CU(cudaMemcpy2DAsync(b, (size_t)ldb * 4, B, (size_t)nb * 4, (size_t)nb * 4, (size_t)rows, cudaMemcpyDeviceToDevice, h->stream));
      h->p.tensor_cores = tensor_cores;
      const int splits = h->gemm_tn(a, lda, b, ldb, ldp, rows, ka, nb);
      h->finish_grad(splits, ka, nb, ldp, c, nullptr, 0, nullptr, nullptr, false);
      h->p.tensor_cores = saved;
      CU(cudaMemcpy2DAsync(C, (size_t)nb * 4, c, (size_t)ldp * 4, (size_t)nb * 4, (size_t)ka, cudaMemcpyDeviceToDevice, h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } catch (...) {
      h->p.tensor_cores = saved;
      cudaFree(a); cudaFree(b); cudaFree(c);
      throw;
    }
    cudaFree(a); cudaFree(b); cudaFree(c);
    h->check_status();
  });
}

// ---- propagation for callers that may not allocate ---------------------------------------------
int gcn_admm_propagate_static(gcn_admm* h, const float* x, int width, float* out) {
  return guarded(h, [&] {
    constexpr long long kStaticElems = 4LL << 20;
    if (!x || !out || width < 1 || width > kMaxWidth) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    if ((long long)h->n * ldpad(width) > kStaticElems)
      throw Fail{GCN_ADMM_ERR_ARG, "n * padded width exceeds the limit of 4194304 floats of this entry point"};
    if (!is_device_pointer(x) || !is_device_pointer(out))
      throw Fail{GCN_ADMM_ERR_ARG, "x and out must be device pointers"};
    struct Untimed {   // event creation reserves memory: launches here are counted, never timed
      gcn_admm* h; bool saved;
      explicit Untimed(gcn_admm* h_) : h(h_), saved(h_->profiling) { h->profiling = false; }
      ~Untimed() { h->profiling = saved; }
    } untimed(h);
    h->propagate_dense(x, width, out, false);
  });
}

int gcn_admm_index(gcn_admm* h, int which, int comm, const int** data, long long* len) {
  return guarded(h, [&] {
    if (!data || !len || which < 0 || which > GCN_ADMM_IX_SEG_BEGIN) throw Fail{GCN_ADMM_ERR_ARG, "bad selector"};
    const GraphIndex& g = h->gi;
    auto give = [&](const auto& v) { *data = v.data(); *len = (long long)v.size(); };
    switch (which) {
      case GCN_ADMM_IX_PERM: give(g.perm); break;
      case GCN_ADMM_IX_INV_PERM: give(g.inv); break;
      case GCN_ADMM_IX_COMM_PTR: give(g.comm_ptr); break;
      case GCN_ADMM_IX_CSR_ROW_PTR: give(g.row_ptr); break;
      case GCN_ADMM_IX_CSR_COL: give(g.col); break;
      case GCN_ADMM_IX_SEG_ROW_PTR: give(g.seg_row_ptr); break;
      case GCN_ADMM_IX_SEG_COMM: give(g.seg_comm); break;
      case GCN_ADMM_IX_SEG_BEGIN: give(g.seg_begin); break;
      default: {
        if (comm < 0 || comm >= h->M) throw Fail{GCN_ADMM_ERR_ARG, "community out of range"};
        std::vector<int>& c = h->ix_cache[which];
        if (which == GCN_ADMM_IX_NBR) c = gcn_admm_host::nbr_of(g, comm);
        else if (which == GCN_ADMM_IX_HALO1) c = gcn_admm_host::halo1_of(g, comm);
        else c = gcn_admm_host::halo2_of(g, comm);
        give(c);
      }
    }
  });
}

namespace {
void ensure_shard_plan(gcn_admm* h, int n_ranks) {
  if (h->shard_plan.n_ranks == n_ranks) return;
  if (!gcn_admm_host::build_shard_plan(h->gi, n_ranks, h->shard_plan))
    throw Fail{GCN_ADMM_ERR_ARG, "n_ranks must be between 1 and the number of communities"};
  h->shard_ranges = h->shard_plan.comm_begin;
  h->shard_ranges.insert(h->shard_ranges.end(), h->shard_plan.row_begin.begin(), h->shard_plan.row_begin.end());
}
}  // namespace

int gcn_admm_shard_plan(gcn_admm* h, int n_ranks, int which, int receiver, int sender, const int** data, long long* len) {
  return guarded(h, [&] {
    if (!data || !len || which < GCN_ADMM_SHARD_RANGES || which > GCN_ADMM_SHARD_SECOND_ORDER)
      throw Fail{GCN_ADMM_ERR_ARG, "bad selector"};
    ensure_shard_plan(h, n_ranks);
    const std::vector<int>* v = &h->shard_ranges;
    if (which != GCN_ADMM_SHARD_RANGES) {
      if (receiver < 0 || receiver >= n_ranks || sender < 0 || sender >= n_ranks)
        throw Fail{GCN_ADMM_ERR_ARG, "rank out of range"};
      const auto& lists = which == GCN_ADMM_SHARD_FIRST_ORDER ? h->shard_plan.first_order : h->shard_plan.second_order;
      v = &lists[(size_t)receiver * n_ranks + sender];
    }
    *data = v->data();
    *len = (long long)v->size();
  });
}

// The propagation as the ranks of a sharded run would carry it out, rank after rank on this one device.
int gcn_admm_propagate_sharded(gcn_admm* h, int n_ranks, const float* x, int width, float* out, long long* staged_rows) {
  return guarded(h, [&] {
    if (!x || !out || width < 1 || width > kMaxWidth) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    ensure_shard_plan(h, n_ranks);
    const gcn_admm_host::ShardPlan& plan = h->shard_plan;
    const gcn_admm_host::GraphIndex& g = h->gi;
    const int ldw = ldpad(width), R = n_ranks;
    const size_t rows = (size_t)h->n;
    const bool dev_in = is_device_pointer(x), dev_out = is_device_pointer(out);
    if (dev_in != dev_out) throw Fail{GCN_ADMM_ERR_ARG, "x and out must both be host or both be device pointers"};
    // Long rows are cut into the items of the unsharded kernel, so that every row is the same sum.
    gcn_admm_host::LongRowTables lt;
    gcn_admm_host::build_long_row_tables(g, h->long_len, lt);
    std::vector<void*> mine;   // freed on every way out
    auto take = [&](size_t bytes) { void* q = dalloc<char>(std::max<size_t>(bytes, 16)); mine.push_back(q); return q; };
    auto release = [&] { for (void* q : mine) cudaFree(q); mine.clear(); };
    long long staged = 0;
    try {
      float* dense = static_cast<float*>(take(rows * width * sizeof(float)));
      float* a = static_cast<float*>(take(rows * ldw * sizeof(float)));
      float* b = static_cast<float*>(take(rows * ldw * sizeof(float)));
      CU(cudaMemcpyAsync(dense, x, rows * width * sizeof(float), dev_in ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                         h->stream));
      gk::k_permute_rows<<<h->grid_for(h->n * ldw), 256, 0, h->stream>>>(dense, a, h->d_inv, h->n, width, ldw, 1);
      CU(cudaGetLastError());
      for (int r = 0; r < R; ++r) {
        const int lo = plan.row_begin[r], hi = plan.row_begin[r + 1], n_own = hi - lo;
        // rows this rank holds: its own, then the first-order rows of every sender (ascending in new ids,
        // because senders own ascending row ranges)
        std::vector<int> held((size_t)n_own);
        for (int i = 0; i < n_own; ++i) held[(size_t)i] = lo + i;
        for (int sdr = 0; sdr < R; ++sdr) {
          const std::vector<int>& f = plan.first_order[(size_t)r * R + sdr];
          held.insert(held.end(), f.begin(), f.end());
        }
        const int n_held = (int)held.size();
        staged += n_held - n_own;
        // local tables: the rank's rows of A + I with columns renumbered to positions in `held`, entry order kept
        std::vector<int> rp((size_t)n_own + 1), order((size_t)n_own);
        const long long e0 = g.row_ptr[lo], e1 = g.row_ptr[hi];
        std::vector<int> cl((size_t)(e1 - e0));
        std::vector<float> dv((size_t)n_held);
        for (int k = 0; k < n_held; ++k) dv[(size_t)k] = g.dinv[(size_t)held[(size_t)k]];
        for (int i = 0; i <= n_own; ++i) rp[(size_t)i] = (int)(g.row_ptr[lo + i] - e0);
        for (long long e = e0; e < e1; ++e) {
          const int j = g.col[(size_t)e];
          int local;
          if (j >= lo && j < hi) local = j - lo;
          else {
            const auto it = std::lower_bound(held.begin() + n_own, held.end(), j);
            if (it == held.end() || *it != j) throw Fail{GCN_ADMM_ERR_CUDA, "plan misses a neighbour row"};
            local = (int)(it - held.begin());
          }
          cl[(size_t)(e - e0)] = local;
        }
        for (int i = 0; i < n_own; ++i) order[(size_t)i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int p_, int q_) { return rp[p_ + 1] - rp[p_] > rp[q_ + 1] - rp[q_]; });
        std::vector<int4> table((size_t)n_own);
        for (int i = 0; i < n_own; ++i) {
          const int r_ = order[(size_t)i];
          int bits;
          std::memcpy(&bits, &dv[(size_t)r_], sizeof bits);
          table[(size_t)i] = make_int4(r_, rp[r_], rp[r_ + 1], bits);
        }
        // the rank's long rows, and their items behind one another
        const auto below = [](const gcn_admm_host::Quad& q, int row) { return q.x < row; };
        const auto row_lo = std::lower_bound(lt.rows.begin(), lt.rows.end(), lo, below), row_hi = std::lower_bound(row_lo, lt.rows.end(), hi, below);
        const int first_item = row_lo < row_hi ? row_lo->y : 0;
        std::vector<int4> items, long_rows;
        std::vector<int> item_row;
        for (auto it = row_lo; it < row_hi; ++it) {
          for (int k = it->y; k < it->y + it->z; ++k) {
            const gcn_admm_host::Quad& q = lt.items[(size_t)k];
            items.push_back(make_int4(q.x - lo, (int)(q.y - e0), (int)(q.z - e0), -1));
            item_row.push_back((int)long_rows.size());
          }
          long_rows.push_back(make_int4(it->x - lo, it->y - first_item, it->z, 0));
        }
        const int n_items = (int)items.size(), n_long = (int)long_rows.size();
        int4* d_items = static_cast<int4*>(take(items.size() * sizeof(int4)));
        int4* d_long = static_cast<int4*>(take(long_rows.size() * sizeof(int4)));
        int* d_item_row = static_cast<int*>(take(item_row.size() * sizeof(int)));
        int* d_done = static_cast<int*>(take(long_rows.size() * sizeof(int)));
        float* item_sums = static_cast<float*>(take(items.size() * ldw * sizeof(float)));
        if (n_items > 0) {
          CU(cudaMemcpyAsync(d_items, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice, h->stream));
          CU(cudaMemcpyAsync(d_long, long_rows.data(), long_rows.size() * sizeof(int4), cudaMemcpyHostToDevice, h->stream));
          CU(cudaMemcpyAsync(d_item_row, item_row.data(), item_row.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
          CU(cudaMemsetAsync(d_done, 0, long_rows.size() * sizeof(int), h->stream));
        }
        int* d_rp = static_cast<int*>(take(rp.size() * sizeof(int)));
        int* d_cl = static_cast<int*>(take(cl.size() * sizeof(int)));
        int4* d_table = static_cast<int4*>(take(table.size() * sizeof(int4)));
        int* d_held = static_cast<int*>(take(held.size() * sizeof(int)));
        float* d_dv = static_cast<float*>(take(dv.size() * sizeof(float)));
        float* xl = static_cast<float*>(take((size_t)n_held * ldw * sizeof(float)));
        CU(cudaMemcpyAsync(d_rp, rp.data(), rp.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
        if (!cl.empty()) CU(cudaMemcpyAsync(d_cl, cl.data(), cl.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
        if (n_own > 0) CU(cudaMemcpyAsync(d_table, table.data(), table.size() * sizeof(int4), cudaMemcpyHostToDevice, h->stream));
        if (n_held > 0) {
          CU(cudaMemcpyAsync(d_held, held.data(), held.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
          CU(cudaMemcpyAsync(d_dv, dv.data(), dv.size() * sizeof(float), cudaMemcpyHostToDevice, h->stream));
          // own rows and, behind them, the copies of the first-order rows: on several devices the second part
          // is what the receives from the rows' owners fill
          gk::k_gather_rows<<<h->grid_for((long long)n_held * (ldw / 4)), 256, 0, h->stream>>>(
              reinterpret_cast<const float4*>(a), d_held, reinterpret_cast<float4*>(xl), ldw / 4, n_held);
          CU(cudaGetLastError());
          ++h->launches;
        }
        if (n_own > 0) {
          gcn_admm::Scope sc(h, "spmm.sharded", 1, 0.0, 0.0);
          h->spmm_tables<4, false>(gcn_admm::GatherGraph{d_rp, d_cl, nullptr, nullptr, d_dv, d_table, d_items, d_long, d_item_row, d_done, n_own, n_items, n_long, h->long_len, item_sums},
                         xl, b + (size_t)lo * ldw, ldw / 4);
        }
        CU(cudaStreamSynchronize(h->stream));   // the host vectors of this rank go out of scope
      }
      gk::k_permute_rows<<<h->grid_for(h->n * ldw), 256, 0, h->stream>>>(b, dense, h->d_inv, h->n, width, ldw, 0);
      CU(cudaGetLastError());
      h->launches += 2;   // the two row permutations
      CU(cudaMemcpyAsync(out, dense, rows * width * sizeof(float), dev_out ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                         h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } catch (...) {
      release();
      throw;
    }
    release();
    if (staged_rows) *staged_rows = staged;
  });
}

int gcn_admm_get_state(gcn_admm* h, int which, int layer, void* out) {
  return guarded(h, [&] {
    if (!out) throw Fail{GCN_ADMM_ERR_ARG, "NULL output"};
    const int L = h->L;
    auto need_layer = [&](int lo, int hi) {
      if (layer < lo || layer > hi) throw Fail{GCN_ADMM_ERR_ARG, "layer out of range"};
    };
    if (which == GCN_ADMM_ST_W) {
      need_layer(1, L);
      const int r = h->C[layer - 1], c = h->C[layer], ldw = h->ld[layer];
      CU(h->stage.get(out, h->W[layer], sizeof(float) * c, sizeof(float) * ldw, r, h->stream));
    } else if (which == GCN_ADMM_ST_Z) {
      need_layer(1, L);
      h->rows_to_host(h->Z[layer], h->C[layer], static_cast<float*>(out));
    } else if (which == GCN_ADMM_ST_U) {
      h->rows_to_host(h->U, h->C[L], static_cast<float*>(out));
    } else if (which == GCN_ADMM_ST_TAU) {
      need_layer(1, L);
      h->take_steps(h->ctl_w + layer, static_cast<double*>(out), 1);
    } else if (which == GCN_ADMM_ST_THETA) {
      need_layer(1, L - 1);
      h->take_steps(h->ctl_z + (size_t)layer * h->M, static_cast<double*>(out), h->M);
    } else if (which == GCN_ADMM_ST_PIPELINE_FLAG) {
      CU(cudaMemcpyAsync(out, h->tc_error, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } else {
      throw Fail{GCN_ADMM_ERR_ARG, "unknown state selector"};
    }
  });
}

int gcn_admm_set_state(gcn_admm* h, int which, int layer, const void* in) {
  return guarded(h, [&] {
    if (!in) throw Fail{GCN_ADMM_ERR_ARG, "NULL input"};
    const int L = h->L;
    auto need_layer = [&](int lo, int hi) {
      if (layer < lo || layer > hi) throw Fail{GCN_ADMM_ERR_ARG, "layer out of range"};
    };
    if (which == GCN_ADMM_ST_W) {
      need_layer(1, L);
      h->upload_weight(layer, static_cast<const float*>(in));
      h->fresh = false;
    } else if (which == GCN_ADMM_ST_Z) {
      need_layer(1, L);
      h->rows_from_host(static_cast<const float*>(in), h->C[layer], h->Z[layer]);
      h->fresh = false;
    } else if (which == GCN_ADMM_ST_U) {
      h->rows_from_host(static_cast<const float*>(in), h->C[L], h->U);
    } else if (which == GCN_ADMM_ST_TAU) {
      need_layer(1, L);
      const double t = *static_cast<const double*>(in);
      if (!(t > 0.0)) throw Fail{GCN_ADMM_ERR_ARG, "tau must be positive"};
      h->put_steps(h->ctl_w + layer, &t, 1);
    } else if (which == GCN_ADMM_ST_THETA) {
      need_layer(1, L - 1);
      const double* t = static_cast<const double*>(in);
      for (int m = 0; m < h->M; ++m)
        if (!(t[m] > 0.0)) throw Fail{GCN_ADMM_ERR_ARG, "theta must be positive"};
      h->put_steps(h->ctl_z + (size_t)layer * h->M, t, h->M);
    } else if (which == GCN_ADMM_ST_PIPELINE_FLAG) {
      CU(cudaMemcpyAsync(h->tc_error, in, sizeof(int), cudaMemcpyHostToDevice, h->stream));
      CU(cudaStreamSynchronize(h->stream));
    } else {
      throw Fail{GCN_ADMM_ERR_ARG, "unknown state selector"};
    }
  });
}

int gcn_admm_launches(gcn_admm* h, long long* count) {
  return guarded(h, [&] {
    if (!count) throw Fail{GCN_ADMM_ERR_ARG, "NULL output"};
    *count = h->launches;
  });
}

int gcn_admm_profile(gcn_admm* h, int enable) {
  return guarded(h, [&] {
    h->collect_profile();
    if (enable) h->prof.clear();
    h->profiling = enable != 0;
  });
}

int gcn_admm_profile_read(gcn_admm* h, int max_entries, int* n_entries, char* names, long long* launches, double* ms,
                          double* bytes, double* flops) {
  return guarded(h, [&] {
    if (!n_entries || max_entries < 0) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    h->collect_profile();
    int k = 0;
    for (const auto& kv : h->prof) {
      if (k >= max_entries) break;
      if (names) { std::strncpy(names + (size_t)k * 48, kv.first.c_str(), 47); names[(size_t)k * 48 + 47] = 0; }
      if (launches) launches[k] = kv.second.launches;
      if (ms) ms[k] = kv.second.ms;
      if (bytes) bytes[k] = kv.second.bytes;
      if (flops) flops[k] = kv.second.flops;
      ++k;
    }
    *n_entries = k;
  });
}

int gcn_admm_decisions(gcn_admm* h, int max_passes, int* n_passes, int* trial_w, double* q_w, int* trial_z,
                       double* q_z) {
  return guarded(h, [&] {
    if (!n_passes || max_passes < 0) throw Fail{GCN_ADMM_ERR_ARG, "bad argument"};
    const int L = h->L;
    const long long have = std::min<long long>(h->log_count, kLogPasses);
    const int take = (int)std::min<long long>(have, max_passes);
    const size_t zper = (size_t)std::max(L - 1, 0) * h->M;
    CU(cudaStreamSynchronize(h->stream));
    for (int k = 0; k < take; ++k) {
      const long long pass = h->log_count - have + k;   // oldest kept pass first
      const long long slot = pass % kLogPasses;
      if (trial_w) CU(cudaMemcpy(trial_w + (size_t)k * L, h->log_trial_w + slot * L, L * sizeof(int), cudaMemcpyDeviceToHost));
      if (q_w) CU(cudaMemcpy(q_w + (size_t)k * L, h->log_q_w + slot * L, L * sizeof(double), cudaMemcpyDeviceToHost));
      if (zper && trial_z)
        CU(cudaMemcpy(trial_z + k * zper, h->log_trial_z + slot * zper, zper * sizeof(int), cudaMemcpyDeviceToHost));
      if (zper && q_z) CU(cudaMemcpy(q_z + k * zper, h->log_q_z + slot * zper, zper * sizeof(double), cudaMemcpyDeviceToHost));
    }
    *n_passes = take;
    h->check_status();
  });
}

}  // extern "C"
