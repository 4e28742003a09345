// Memory of a handle: one device slab that all its matrices and tables are cut from, and a page-locked staging
// buffer through which host buffers are copied in both directions.
//
// A handle has about sixty device buffers.  Allocated one by one they cost 5 ms to create and 2 ms to free on a quiet
// machine, more than the twenty passes of a small training run, and ten times that where other processes use the
// driver too.  create and destroy of a handle of 2.7 k nodes, 1433-16-7: 1.6 ms on memory an earlier handle left, 8 to 15
// without (slab, 12 MB of page-locked memory), 26 as the first of a process; 169 k nodes, 128-256-256-40: 14, 22 to 29, 45.
// Copies between the device and pageable host memory go through the driver's own staging on one core at
// 5-10 GB/s; here several cores fill or drain one part of the staging buffer while the copy engine works on the next.
//
// Slabs, staging buffers and streams of destroyed handles are kept for later ones up to a fixed amount (kIdleSlabBytes,
// kIdleStages; the oldest go first), under a lock, and only after the work that used them has finished; the rest goes back
// to the driver at once, the idle slabs of a device when an allocation of the library fails there, and everything when the
// caller asks for it (gcn_admm_release_idle) and at exit.
#pragma once
#include <cuda_runtime.h>
#include <omp.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

namespace gcn_admm_mem {

constexpr std::size_t kIdleSlabBytes = (std::size_t)3 << 30;     // device memory kept for later handles, all devices together
constexpr std::size_t kIdleStages = 4;
constexpr std::size_t kSlot = (std::size_t)4 << 20;               // a staging buffer is kSlots parts of this size
constexpr int kSlots = 3;

struct Slab {
  int device = 0;
  char* base = nullptr;
  std::size_t size = 0;
};

class Pool {
 public:
  static Pool& get() {
    static Pool pool;
    return pool;
  }
  // A slab of at least `bytes` on the current device (`device`).
  cudaError_t take(int device, std::size_t bytes, Slab* out) {
    const std::size_t grain = (std::size_t)2 << 20;
    bytes = (bytes + grain - 1) / grain * grain;
    {
      std::lock_guard<std::mutex> lock(mutex_);
      auto best = idle_.end();
      for (auto it = idle_.begin(); it != idle_.end(); ++it)
        if (it->device == device && it->size >= bytes && it->size <= 2 * bytes + 8 * grain && (best == idle_.end() || it->size < best->size))
          best = it;
      if (best != idle_.end()) {
        *out = *best;
        idle_bytes_ -= best->size;
        idle_.erase(best);
        return cudaSuccess;
      }
    }
    void* p = nullptr;
    const cudaError_t e = allocate(device, bytes, &p);
    if (e == cudaSuccess) *out = Slab{device, static_cast<char*>(p), bytes};
    return e;
  }
  // cudaMalloc on the current device (`device`); where that fails, once more without the idle slabs.
  cudaError_t allocate(int device, std::size_t bytes, void** out) {
    cudaError_t e = cudaMalloc(out, bytes);
    if (e == cudaErrorMemoryAllocation && release_slabs(device)) {
      cudaGetLastError();
      e = cudaMalloc(out, bytes);
    }
    return e;
  }
  // What follows is called where a handle ends and throws nothing: what cannot be noted down for keeping is freed.
  // The slab's device is current and no work uses the slab any more.
  void give(const Slab& s) noexcept {
    if (!s.base) return;
    for (;;) {   // the oldest make room; their work has finished too
      Slab oldest;
      {
        std::lock_guard<std::mutex> lock(mutex_);
        if (s.size > kIdleSlabBytes) break;
        if (idle_bytes_ + s.size <= kIdleSlabBytes) {
          if (!note(idle_, s)) break;
          idle_bytes_ += s.size;
          return;
        }
        oldest = idle_.front();
        idle_bytes_ -= oldest.size;
        idle_.erase(idle_.begin());
      }
      cudaFree(oldest.base);
    }
    cudaFree(s.base);
  }
  char* take_stage() {
    {
      std::lock_guard<std::mutex> lock(mutex_);
      if (!stages_.empty()) {
        char* p = stages_.back();
        stages_.pop_back();
        return p;
      }
    }
    void* p = nullptr;
    if (cudaHostAlloc(&p, kSlot * kSlots, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return static_cast<char*>(p);
  }
  void give_stage(char* p) noexcept {
    if (!p) return;
    {
      std::lock_guard<std::mutex> lock(mutex_);
      if (stages_.size() < kIdleStages && note(stages_, p)) return;
    }
    cudaFreeHost(p);
  }
  // A non-blocking stream of the current device (`device`); given back when nothing is in flight on it.
  cudaError_t take_stream(int device, cudaStream_t* out) {
    {
      std::lock_guard<std::mutex> lock(mutex_);
      for (auto it = streams_.begin(); it != streams_.end(); ++it)
        if (it->first == device) {
          *out = it->second;
          streams_.erase(it);
          return cudaSuccess;
        }
    }
    return cudaStreamCreateWithFlags(out, cudaStreamNonBlocking);
  }
  void give_stream(int device, cudaStream_t s) noexcept {
    {
      std::lock_guard<std::mutex> lock(mutex_);
      if (streams_.size() < kIdleStages && note(streams_, std::make_pair(device, s))) return;
    }
    cudaStreamDestroy(s);
  }
  // Gives everything idle back to the driver.
  void release() noexcept {
    release_slabs(kAnyDevice);
    std::vector<char*> stages;
    std::vector<std::pair<int, cudaStream_t>> streams;
    {
      std::lock_guard<std::mutex> lock(mutex_);
      stages.swap(stages_);
      streams.swap(streams_);
    }
    for (char* p : stages) cudaFreeHost(p);
    for (const auto& s : streams) cudaStreamDestroy(s.second);
  }
  ~Pool() { release(); }   // at exit the driver may already be gone: its error is of no consequence then

 private:
  static constexpr int kAnyDevice = -1;
  // Whether there was anything to give back.
  bool release_slabs(int device) noexcept {
    for (bool any = false;; any = true) {
      Slab s;
      {
        std::lock_guard<std::mutex> lock(mutex_);
        const auto it = std::find_if(idle_.begin(), idle_.end(), [&](const Slab& q) { return device == kAnyDevice || q.device == device; });
        if (it == idle_.end()) return any;
        s = *it;
        idle_bytes_ -= s.size;
        idle_.erase(it);
      }
      cudaFree(s.base);
    }
  }
  template <typename T>
  static bool note(std::vector<T>& list, const T& x) noexcept {
    try { list.push_back(x); return true; } catch (const std::bad_alloc&) { return false; }
  }
  std::mutex mutex_;
  std::vector<Slab> idle_;
  std::size_t idle_bytes_ = 0;
  std::vector<char*> stages_;
  std::vector<std::pair<int, cudaStream_t>> streams_;
};

// memcpy by several threads where it pays (a core moves about 10 GB/s, less into pages that are touched first here): at most
// eight, and no more than the caller allows OpenMP (OMP_NUM_THREADS, omp_set_num_threads).
inline void copy_bytes(void* dst, const void* src, std::size_t bytes) {
  constexpr std::size_t kPiece = (std::size_t)256 << 10;
  if (bytes < 4 * kPiece) { std::memcpy(dst, src, bytes); return; }
  const long long pieces = (long long)((bytes + kPiece - 1) / kPiece);
#pragma omp parallel for schedule(static) num_threads(std::min(8, omp_get_max_threads()))
  for (long long i = 0; i < pieces; ++i) {
    const std::size_t at = (std::size_t)i * kPiece;
    std::memcpy(static_cast<char*>(dst) + at, static_cast<const char*>(src) + at, std::min(kPiece, bytes - at));
  }
}

// Is `p` host memory the copy engine can reach by itself (page-locked)?
inline bool page_locked(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return false; }
  return a.type == cudaMemoryTypeHost;
}

// The staging buffer of one handle.  Copies are enqueued on the handle's stream; kSlots parts take turns, each with an
// event after its last use.
class Stage {
 public:
  cudaError_t open() {
    if (base_) return cudaSuccess;
    base_ = Pool::get().take_stage();
    if (!base_) return cudaErrorMemoryAllocation;
    for (cudaEvent_t& e : used_) {
      const cudaError_t err = cudaEventCreateWithFlags(&e, cudaEventDisableTiming);
      if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
  }
  // Nothing is in flight any more.
  void close() {
    for (cudaEvent_t& e : used_)
      if (e) { cudaEventDestroy(e); e = nullptr; }
    Pool::get().give_stage(base_);
    base_ = nullptr;
  }

  // Host -> device.  Small pieces whose destinations follow each other (up to `slack` bytes apart) leave as one copy; flush()
  // sends the last one.  The source may be reused after finish().
  cudaError_t put(void* dst, const void* src, std::size_t bytes, cudaStream_t stream) {
    if (bytes == 0) return cudaSuccess;
    if (bytes >= kSlot / 4 && page_locked(src)) {
      if (const cudaError_t e = flush(stream)) return e;
      direct_ = true;
      return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, stream);
    }
    constexpr std::ptrdiff_t slack = 256;
    char* d = static_cast<char*>(dst);
    const char* s = static_cast<const char*>(src);
    while (bytes > 0) {
      const std::ptrdiff_t gap = d - (run_dst_ + run_);
      if (run_ == 0 || gap < 0 || gap > slack || run_ + (std::size_t)gap >= kSlot) {
        if (const cudaError_t e = flush(stream)) return e;
        if (const cudaError_t e = cudaEventSynchronize(used_[slot_])) return e;
        run_dst_ = d;
      } else if (gap > 0) {
        std::memset(part() + run_, 0, (std::size_t)gap);   // alignment gap between two tables of the slab
        run_ += (std::size_t)gap;
      }
      const std::size_t now = std::min(bytes, kSlot - run_);
      copy_bytes(part() + run_, s, now);
      run_ += now; d += now; s += now; bytes -= now;
      if (run_ == kSlot)
        if (const cudaError_t e = flush(stream)) return e;
    }
    return cudaSuccess;
  }
  // Ends an upload: sends what is left and waits where a source is still being read in place.
  cudaError_t finish(cudaStream_t stream) {
    if (const cudaError_t e = flush(stream)) return e;
    if (!direct_) return cudaSuccess;
    direct_ = false;
    return cudaStreamSynchronize(stream);
  }
  cudaError_t flush(cudaStream_t stream) {
    if (run_ == 0) return cudaSuccess;
    cudaError_t e = cudaMemcpyAsync(run_dst_, part(), run_, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaEventRecord(used_[slot_], stream);
    run_ = 0;
    slot_ = (slot_ + 1) % kSlots;
    return e;
  }

  // A part of the buffer that kernels may read (after the host has filled it) or write: valid until leave().
  // At most kSlot bytes.
  cudaError_t enter(cudaStream_t stream, char** out) {
    if (const cudaError_t e = flush(stream)) return e;
    if (const cudaError_t e = cudaEventSynchronize(used_[slot_])) return e;
    *out = part();
    return cudaSuccess;
  }
  cudaError_t leave(cudaStream_t stream) {
    const cudaError_t e = cudaEventRecord(used_[slot_], stream);
    slot_ = (slot_ + 1) % kSlots;
    return e;
  }

  // Device -> host: `count` dense arrays one after the other, the bus moving on to the next while the host still empties the parts of
  // the one before.  Returns with the host buffers filled.
  struct Part {
    void* dst;
    const void* src;
    std::size_t bytes;
  };
  cudaError_t get_all(const Part* parts, int count, cudaStream_t stream) {
    if (const cudaError_t e = flush(stream)) return e;
    bool direct = false;
    int p_begun = 0, p_done = 0;             // array and offset of the next piece to start and of the next to empty
    std::size_t at_begun = 0, at_done = 0, begun = 0, done = 0;
    const auto staged = [&](int p) { return parts[p].bytes > 0 && !(parts[p].bytes >= kSlot / 4 && page_locked(parts[p].dst)); };
    for (int p = 0; p < count; ++p)
      if (parts[p].bytes > 0 && !staged(p)) {
        direct = true;
        if (const cudaError_t e = cudaMemcpyAsync(parts[p].dst, parts[p].src, parts[p].bytes, cudaMemcpyDeviceToHost, stream)) return e;
      }
    const auto skip = [&](int& p) { while (p < count && !staged(p)) ++p; };
    skip(p_begun);
    skip(p_done);
    while (p_done < count) {
      while (p_begun < count && begun < done + kSlots) {
        const std::size_t k = (slot_ + begun) % kSlots, len = std::min(kSlot, parts[p_begun].bytes - at_begun);
        cudaError_t e = cudaEventSynchronize(used_[k]);
        if (e == cudaSuccess) e = cudaMemcpyAsync(base_ + k * kSlot, static_cast<const char*>(parts[p_begun].src) + at_begun, len, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaEventRecord(used_[k], stream);
        if (e != cudaSuccess) return e;
        ++begun;
        at_begun += len;
        if (at_begun == parts[p_begun].bytes) { at_begun = 0; ++p_begun; skip(p_begun); }
      }
      const std::size_t k = (slot_ + done) % kSlots, len = std::min(kSlot, parts[p_done].bytes - at_done);
      if (const cudaError_t e = cudaEventSynchronize(used_[k])) return e;
      copy_bytes(static_cast<char*>(parts[p_done].dst) + at_done, base_ + k * kSlot, len);
      ++done;
      at_done += len;
      if (at_done == parts[p_done].bytes) { at_done = 0; ++p_done; skip(p_done); }
    }
    slot_ = (int)((slot_ + done) % kSlots);
    return direct ? cudaStreamSynchronize(stream) : cudaSuccess;
  }

  // Device -> host: `rows` rows of `width` bytes, `pitch` bytes apart on the device, dense on the host.  Returns with the
  // host buffer filled.
  cudaError_t get(void* dst, const void* src, std::size_t width, std::size_t pitch, std::size_t rows, cudaStream_t stream) {
    if (width == 0 || rows == 0) return cudaSuccess;
    if (const cudaError_t e = flush(stream)) return e;
    if (width == pitch) { width *= rows; pitch = width; rows = 1; }
    if (width * rows >= kSlot / 4 && page_locked(dst)) {
      const cudaError_t e = rows == 1 ? cudaMemcpyAsync(dst, src, width, cudaMemcpyDeviceToHost, stream)
                                      : cudaMemcpy2DAsync(dst, width, src, pitch, width, rows, cudaMemcpyDeviceToHost, stream);
      return e ? e : cudaStreamSynchronize(stream);
    }
    // pieces of at most a slot: whole rows, or parts of one row when a row is longer than that
    const std::size_t rows_at_once = std::max<std::size_t>(1, kSlot / width);
    const std::size_t per_row = rows == 1 ? (width + kSlot - 1) / kSlot : 1;
    if (rows > 1 && width > kSlot) {
      for (std::size_t r = 0; r < rows; ++r)
        if (const cudaError_t e = get(static_cast<char*>(dst) + r * width, static_cast<const char*>(src) + r * pitch, width, width, 1, stream)) return e;
      return cudaSuccess;
    }
    const std::size_t pieces = rows == 1 ? per_row : (rows + rows_at_once - 1) / rows_at_once;
    auto begin = [&](std::size_t i) -> cudaError_t {
      char* to = base_ + (std::size_t)((slot_ + i) % kSlots) * kSlot;
      cudaError_t e = cudaEventSynchronize(used_[(slot_ + i) % kSlots]);
      if (e != cudaSuccess) return e;
      if (rows == 1) e = cudaMemcpyAsync(to, static_cast<const char*>(src) + i * kSlot, std::min(kSlot, width - i * kSlot), cudaMemcpyDeviceToHost, stream);
      else e = cudaMemcpy2DAsync(to, width, static_cast<const char*>(src) + i * rows_at_once * pitch, pitch, width,
                                 std::min(rows_at_once, rows - i * rows_at_once), cudaMemcpyDeviceToHost, stream);
      return e ? e : cudaEventRecord(used_[(slot_ + i) % kSlots], stream);
    };
    for (std::size_t i = 0; i < std::min<std::size_t>(pieces, kSlots - 1); ++i)
      if (const cudaError_t e = begin(i)) return e;
    for (std::size_t i = 0; i < pieces; ++i) {
      if (i + kSlots - 1 < pieces)
        if (const cudaError_t e = begin(i + kSlots - 1)) return e;
      if (const cudaError_t e = cudaEventSynchronize(used_[(slot_ + i) % kSlots])) return e;
      const std::size_t at = rows == 1 ? i * kSlot : i * rows_at_once * width;
      const std::size_t len = rows == 1 ? std::min(kSlot, width - at) : std::min(rows_at_once, rows - i * rows_at_once) * width;
      copy_bytes(static_cast<char*>(dst) + at, base_ + (std::size_t)((slot_ + i) % kSlots) * kSlot, len);
    }
    slot_ = (int)((slot_ + pieces) % kSlots);
    return cudaSuccess;
  }

 private:
  char* part() { return base_ + (std::size_t)slot_ * kSlot; }
  char* base_ = nullptr;
  cudaEvent_t used_[kSlots] = {};
  int slot_ = 0;
  char* run_dst_ = nullptr;   // destination of the run being filled and its length so far
  std::size_t run_ = 0;
  bool direct_ = false;       // a page-locked source is being read by the copy engine
};

}  // namespace gcn_admm_mem
