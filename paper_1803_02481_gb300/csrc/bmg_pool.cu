// Device memory kept between hierarchies.
//
// A setup and solve of a 255^2 problem is 1.0 ms of GPU work, and mapping and
// unmapping its memory took another 0.7 ms (cudaMalloc 0.24, cudaMallocHost
// 0.13, cudaFree 0.2, cudaFreeHost 0.13); at 8191^2 cudaMalloc and cudaFree
// are 4.7 of 92 ms.  A program that assembles such problems anew all the time
// (an outer iteration, a gradient) pays it on every one.  Blocks that a
// hierarchy gives back are therefore kept for the next.
//
//  * Bounded: at most 1/32 of the device's memory is kept per device; the
//    oldest blocks go back to the driver first, and all of them when an
//    allocation fails (and the allocation is tried again) or the caller asks
//    (bmg_release_memory).
//  * A block is kept only if the work on it is done when it is given back (its
//    owner waits for what it left under way, see Pending), so it does not
//    matter which streams used it or will use it; any other goes to cudaFree,
//    which waits for it.
//  * Thread-safe; blocks stay on their device.
#include "bmg_internal.h"

#include <algorithm>
#include <list>
#include <map>
#include <mutex>

namespace bmg {

namespace {

struct Block {
  void* p;
  size_t bytes;
  int dev;
};

struct Pool {
  std::mutex mu;
  std::map<void*, Block> live;
  std::list<Block> kept;               // oldest first
  std::map<int, size_t> kept_bytes;    // per device
  // pinned slots
  std::vector<void*> slots;            // free ones
  std::vector<void*> slabs;
};

// Never destroyed: objects with static lifetime may still give blocks back
// while the process exits.
Pool& pool() {
  static Pool* p = new Pool;
  return *p;
}

constexpr size_t kSlot = 256;          // a pinned slot: the mirror of a solve's scalars
constexpr int kSlabSlots = 64;

size_t keep_limit(int dev) {
  static std::mutex mu;
  static std::map<int, size_t> limits;
  std::lock_guard<std::mutex> g(mu);
  auto it = limits.find(dev);
  if (it != limits.end()) return it->second;
  size_t avail = 0, total = 0;
  if (cudaMemGetInfo(&avail, &total) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return limits[dev] = total / 32;
}

// Returns kept blocks of `dev` to the driver until at most `most` bytes stay.
void trim(Pool& P, int dev, size_t most) {
  for (auto it = P.kept.begin(); it != P.kept.end() && P.kept_bytes[dev] > most;) {
    if (it->dev != dev) {
      ++it;
      continue;
    }
    P.kept_bytes[dev] -= it->bytes;
    cudaFree(it->p);
    it = P.kept.erase(it);
  }
}

cudaError_t malloc_or_trim(Pool& P, int dev, void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    trim(P, dev, 0);
    e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) cudaGetLastError();
  }
  return e;
}

}  // namespace

void* pool_alloc(size_t bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  Pool& P = pool();
  std::lock_guard<std::mutex> g(P.mu);
  // the smallest kept block that fits without wasting more than a quarter
  auto best = P.kept.end();
  for (auto it = P.kept.begin(); it != P.kept.end(); ++it)
    if (it->dev == dev && it->bytes >= bytes && it->bytes - bytes <= bytes / 4 + (size_t(1) << 20) &&
        (best == P.kept.end() || it->bytes < best->bytes))
      best = it;
  if (best != P.kept.end()) {
    const Block b = *best;
    P.kept.erase(best);
    P.kept_bytes[dev] -= b.bytes;
    P.live[b.p] = b;
    return b.p;
  }
  void* p = nullptr;
  if (malloc_or_trim(P, dev, &p, bytes) != cudaSuccess) return nullptr;
  P.live[p] = Block{p, bytes, dev};
  return p;
}

cudaError_t device_malloc(void** p, size_t bytes) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  Pool& P = pool();
  std::lock_guard<std::mutex> g(P.mu);
  return malloc_or_trim(P, dev, p, bytes);
}

Pending::~Pending() {
  for (Entry& e : entries_) cudaEventDestroy(e.done);
}

void Pending::left(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    unknown_ = true;   // runs whenever the caller's graph does
    return;
  }
  for (Entry& e : entries_)
    if (e.stream == s) {
      // (the wait holds nothing up on the stream that recorded the event, and
      // orders a new stream of the same handle behind the old one)
      if (cudaStreamWaitEvent(s, e.done, 0) != cudaSuccess || cudaEventRecord(e.done, s) != cudaSuccess)
        unknown_ = true;
      return;
    }
  Entry e{s, nullptr};
  if (cudaEventCreateWithFlags(&e.done, cudaEventDisableTiming) != cudaSuccess) {
    unknown_ = true;
    return;
  }
  entries_.push_back(e);
  if (cudaEventRecord(e.done, s) != cudaSuccess) unknown_ = true;
}

bool Pending::wait() {
  for (Entry& e : entries_)
    if (cudaEventSynchronize(e.done) != cudaSuccess) unknown_ = true;
  if (unknown_) cudaGetLastError();
  return !unknown_;
}

void pool_free(void* p, bool idle) {
  if (!p) return;
  Pool& P = pool();
  Block b{};
  {
    std::lock_guard<std::mutex> g(P.mu);
    auto it = P.live.find(p);
    if (it == P.live.end()) return;
    b = it->second;
    P.live.erase(it);
  }
  int cur = b.dev;
  cudaGetDevice(&cur);
  if (cur != b.dev) cudaSetDevice(b.dev);
  const size_t limit = keep_limit(b.dev);
  if (!idle || b.bytes > limit) {
    cudaFree(p);
  } else {
    std::lock_guard<std::mutex> g(P.mu);
    trim(P, b.dev, limit - b.bytes);
    P.kept.push_back(b);
    P.kept_bytes[b.dev] += b.bytes;
  }
  if (cur != b.dev) cudaSetDevice(cur);
}

void* pinned_slot(size_t bytes) {
  if (bytes > kSlot) return nullptr;
  Pool& P = pool();
  std::lock_guard<std::mutex> g(P.mu);
  if (P.slots.empty()) {
    void* s = nullptr;
    if (cudaHostAlloc(&s, kSlot * kSlabSlots, cudaHostAllocPortable) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    P.slabs.push_back(s);
    for (int i = kSlabSlots - 1; i >= 0; --i) P.slots.push_back(static_cast<char*>(s) + size_t(i) * kSlot);
  }
  void* p = P.slots.back();
  P.slots.pop_back();
  return p;
}

// (A slab is 16 KB and serves 64 live objects; slabs beyond the first go back
// when no slot is in use.)
void pinned_slot_free(void* p) {
  if (!p) return;
  Pool& P = pool();
  std::lock_guard<std::mutex> g(P.mu);
  P.slots.push_back(p);
  if (P.slabs.size() > 1 && P.slots.size() == P.slabs.size() * kSlabSlots) {
    for (size_t i = 1; i < P.slabs.size(); ++i) cudaFreeHost(P.slabs[i]);
    P.slabs.resize(1);
    P.slots.clear();
    for (int i = kSlabSlots - 1; i >= 0; --i)
      P.slots.push_back(static_cast<char*>(P.slabs[0]) + size_t(i) * kSlot);
  }
}

}  // namespace bmg

extern "C" void bmg_release_memory(void) {
  using namespace bmg;
  Pool& P = pool();
  std::lock_guard<std::mutex> g(P.mu);
  int cur = 0;
  const bool known = cudaGetDevice(&cur) == cudaSuccess;
  for (auto& kept : P.kept_bytes)
    if (kept.second > 0 && cudaSetDevice(kept.first) == cudaSuccess) trim(P, kept.first, 0);
  if (known) cudaSetDevice(cur);
}
