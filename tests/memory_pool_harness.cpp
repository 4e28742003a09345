// Host-only program for test_memory_pool.py: with an argument, the threads of the process after a copy of that many bytes; else the pool of memory.hpp on a stand-in for the CUDA runtime whose device memory is
// a byte count with a limit.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <new>
#include <vector>

#include "memory.hpp"

static std::size_t limit = 0, device_bytes = 0, host_bytes = 0, streams = 0;
static int failures = 0;
static std::map<void*, std::size_t> sizes;

extern "C" {
cudaError_t CUDARTAPI cudaMalloc(void** p, std::size_t bytes) {
  if (device_bytes + bytes > limit) { ++failures; return cudaErrorMemoryAllocation; }
  *p = std::malloc(1);
  sizes[*p] = bytes;
  device_bytes += bytes;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFree(void* p) { device_bytes -= sizes.at(p); sizes.erase(p); std::free(p); return cudaSuccess; }
cudaError_t CUDARTAPI cudaHostAlloc(void** p, std::size_t bytes, unsigned) { *p = std::malloc(1); sizes[*p] = bytes; host_bytes += bytes; return cudaSuccess; }
cudaError_t CUDARTAPI cudaFreeHost(void* p) { host_bytes -= sizes.at(p); sizes.erase(p); std::free(p); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { ++streams; *s = reinterpret_cast<cudaStream_t>(streams); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamDestroy(cudaStream_t) { --streams; return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError() { return cudaSuccess; }
}

static bool no_memory = false;   // every allocation of the host's fails
void* operator new(std::size_t n) {
  void* p = no_memory ? nullptr : std::malloc(n);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

#define NEED(c) \
  if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; }

static int threads_after_copy(std::size_t bytes) {
  std::vector<char> from(bytes, 7), to(bytes);
  gcn_admm_mem::copy_bytes(to.data(), from.data(), bytes);
  int n = -1;
  char line[256];
  std::FILE* f = std::fopen("/proc/self/status", "r");
  while (f && std::fgets(line, sizeof line, f)) std::sscanf(line, "Threads: %d", &n);
  if (f) std::fclose(f);
  return to == from ? n : -1;
}

int main(int argc, char** argv) {
  if (argc > 1) { std::printf("%d\n", threads_after_copy(std::strtoull(argv[1], nullptr, 10))); return 0; }
  using namespace gcn_admm_mem;
  constexpr std::size_t GB = (std::size_t)1 << 30;
  Pool& pool = Pool::get();
  limit = 8 * GB;
  Slab a, b, c;
  NEED(pool.take(0, GB, &a) == cudaSuccess && pool.take(0, 2 * GB, &b) == cudaSuccess && pool.take(1, 2 * GB, &c) == cudaSuccess);
  NEED(device_bytes == 5 * GB);
  pool.give(a);
  pool.give(b);
  NEED(device_bytes == 5 * GB);              // 3 GB idle: the bound
  pool.give(c);                              // the oldest make room: both, with either the bound is passed
  NEED(device_bytes == 2 * GB);
  char* stage[6];
  for (char*& s : stage) s = pool.take_stage();
  for (char* s : stage) pool.give_stage(s);
  cudaStream_t st;
  NEED(pool.take_stream(0, &st) == cudaSuccess);
  pool.give_stream(0, st);
  NEED(host_bytes == kIdleStages * kSlot * kSlots && streams == 1);
  pool.release();                            // all of it goes back
  NEED(device_bytes == 0 && host_bytes == 0 && streams == 0);

  // any allocation of the library that fails takes the idle slabs of its device back, and only those
  limit = 4 * GB;
  NEED(pool.take(0, GB, &a) == cudaSuccess && pool.take(1, GB, &b) == cudaSuccess);
  pool.give(a);
  pool.give(b);
  void* p = nullptr;
  NEED(pool.allocate(0, 3 * GB, &p) == cudaSuccess && failures == 1 && device_bytes == 4 * GB);
  NEED(pool.allocate(0, GB, &p) == cudaErrorMemoryAllocation && failures == 2 && device_bytes == 4 * GB);   // nothing of device 0 is idle: no second try
  NEED(pool.take(1, GB, &c) == cudaSuccess && c.base == b.base);

  // a handle ends without host memory: nothing is thrown, what cannot be kept goes back
  pool.release();
  limit = 8 * GB;
  device_bytes = 0;
  std::vector<Slab> many(64);
  for (Slab& s : many) NEED(pool.take(0, GB / 32, &s) == cudaSuccess);
  stage[0] = pool.take_stage();
  NEED(pool.take_stream(0, &st) == cudaSuccess);
  no_memory = true;
  for (const Slab& s : many) pool.give(s);
  pool.give_stage(stage[0]);
  pool.give_stream(0, st);
  pool.release();
  no_memory = false;
  NEED(device_bytes == 0 && host_bytes == 0 && streams == 0);
  std::printf("ok\n");
  return 0;
}
