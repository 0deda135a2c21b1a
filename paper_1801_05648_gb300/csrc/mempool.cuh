// Device memory: the pools of the set-up calls and the owning buffer.
#pragma once
#include "error.cuh"

#include <cuda_runtime.h>
#include <atomic>
#include <cstddef>
#include <iterator>
#include <map>
#include <memory>
#include <mutex>
#include <set>
#include <utility>
#include <vector>

namespace fsi {

// Device memory that a context keeps between its set-up calls.  A preconditioner build
// makes about a thousand allocations, most of them temporaries of the sizes that the
// build before had; cudaMalloc and cudaFree (which waits for the device) took a third of a
// 256x128 rebuild.  A buffer allocated inside a SetupPhase comes from the context's pool
// and goes back to it when it is released, without waiting: a pool's buffers are only taken for
// work on one stream (the context's, or that of a hierarchy's branch, see precond_build), so a
// block's next user is ordered behind its last one.  A context has five pools (its own and one for each of the
// four branches).  Together they keep at most kKeep bytes of released blocks from one set-up call to the
// next (a rebuild's first act is to release the hierarchies that it is about to build again, so the bound holds
// at the end of a call, see settle), return them when the context is freed, and give them up when any
// allocation of the library fails; an allocator beside the library cannot ask for them.
// Blocks of up to kSmall bytes are cut from slabs that the context's pools share, so that a small
// system's arrays lie in a few large pages and cost no driver call each.  Slabs live as long as
// the context; when kSlabs of them are cut up, a small block is a large one of its own.
class Slabs {
 public:
  static constexpr size_t kSmall = (size_t)1 << 20, kSlab = (size_t)32 << 20;
  static constexpr size_t kSlabs = 8, kKeep = (size_t)1 << 30;
  Slabs() = default;
  Slabs(const Slabs&) = delete;
  Slabs& operator=(const Slabs&) = delete;
  ~Slabs() {
    for (void* p : slabs_) cudaFree(p);
  }
  void* take(size_t bytes);   // null when the slabs are cut up
  // account of the large blocks released to the context's pools
  void hold(size_t bytes) { held_.fetch_add(bytes); }
  void unhold(size_t bytes) { held_.fetch_sub(bytes); }
  size_t held() const { return held_.load(); }

 private:
  std::mutex lock_;
  std::vector<void*> slabs_;
  size_t left_ = 0;
  std::atomic<size_t> held_{0};   // (not under lock_: a slab's allocation may have the pools give up their blocks)
};

class MemPool {
 public:
  explicit MemPool(std::shared_ptr<Slabs> slabs) : slabs_(std::move(slabs)) {
    std::lock_guard<std::mutex> g(registry_lock());
    registry().insert(this);
  }
  ~MemPool() {
    {
      std::lock_guard<std::mutex> g(registry_lock());
      registry().erase(this);
    }
    trim();
  }
  MemPool(const MemPool&) = delete;
  MemPool& operator=(const MemPool&) = delete;

  // at least `bytes` bytes; got: the block's size, to be handed back with it
  void* take(size_t bytes, size_t& got) {
    size_t step = 256;
    while (step * 16 <= bytes && bytes > Slabs::kSmall) step *= 2;   // sizes rounded up by at most an eighth
    bytes = (bytes + step - 1) / step * step;
    {
      std::lock_guard<std::mutex> g(lock_);
      auto it = free_.lower_bound(bytes);
      if (it != free_.end() && it->first <= bytes + bytes / 4 + 4096 &&
          (it->first <= Slabs::kSmall) == (bytes <= Slabs::kSmall)) {
        void* p = it->second;
        got = it->first;
        if (got > Slabs::kSmall) slabs_->unhold(got);
        free_.erase(it);
        return p;
      }
    }
    if (bytes <= Slabs::kSmall) {
      void* p = slabs_->take(bytes);
      if (!p) return take(Slabs::kSmall + 1, got);
      got = bytes;
      return p;
    }
    got = bytes;
    return device_malloc(bytes);
  }
  void give(void* p, size_t bytes) {
    std::lock_guard<std::mutex> g(lock_);
    free_.emplace(bytes, p);
    if (bytes > Slabs::kSmall) slabs_->hold(bytes);
  }
  // frees blocks, the largest first, until the context's pools hold kKeep bytes or this one has none
  void settle() {
    std::lock_guard<std::mutex> g(lock_);
    while (slabs_->held() > Slabs::kKeep && !free_.empty()) {
      auto it = std::prev(free_.end());
      if (it->first <= Slabs::kSmall) break;
      cudaFree(it->second);
      slabs_->unhold(it->first);
      free_.erase(it);
    }
  }
  // frees the blocks held (those of the slabs stay)
  void trim() {
    std::lock_guard<std::mutex> g(lock_);
    auto it = free_.upper_bound(Slabs::kSmall);
    for (auto i = it; i != free_.end(); ++i) {
      cudaFree(i->second);
      slabs_->unhold(i->first);
    }
    free_.erase(it, free_.end());
  }
  // cudaMalloc; when memory is short, once more after every pool has freed what it holds
  static void* device_malloc(size_t bytes) {
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      {
        std::lock_guard<std::mutex> g(registry_lock());
        for (MemPool* q : registry()) q->trim();
      }
      e = cudaMalloc(&p, bytes);
      if (e != cudaSuccess) cudaGetLastError();   // reported here: the next launch's check does not find it again
    }
    FSI_CUDA(e);
    return p;
  }

 private:
  static std::mutex& registry_lock() {
    static auto* m = new std::mutex;
    return *m;
  }
  static std::set<MemPool*>& registry() {
    static auto* r = new std::set<MemPool*>;   // never destroyed: a context may outlive static objects
    return *r;
  }
  std::shared_ptr<Slabs> slabs_;
  std::mutex lock_;
  std::multimap<size_t, void*> free_;
};

inline void* Slabs::take(size_t bytes) {
  std::lock_guard<std::mutex> g(lock_);
  if (slabs_.empty() || left_ < bytes) {
    if (slabs_.size() >= kSlabs) return nullptr;
    slabs_.reserve(slabs_.size() + 1);
    slabs_.push_back(MemPool::device_malloc(kSlab));
    left_ = kSlab;
  }
  void* p = static_cast<char*>(slabs_.back()) + (kSlab - left_);
  left_ -= bytes;
  return p;
}

// The pool that this thread's set-up call allocates from (null outside one).
inline std::shared_ptr<MemPool>& current_pool() {
  thread_local std::shared_ptr<MemPool> p;
  return p;
}

// Owning device buffer.
template <class T>
struct DBuf {
  T* p = nullptr;
  size_t n = 0;
  DBuf() = default;
  explicit DBuf(size_t count) { alloc(count); }
  DBuf(const DBuf&) = delete;
  DBuf& operator=(const DBuf&) = delete;
  DBuf(DBuf&& o) noexcept : p(o.p), n(o.n), pool(std::move(o.pool)), bytes(o.bytes) { o.p = nullptr; o.n = 0; }
  DBuf& operator=(DBuf&& o) noexcept {
    if (this != &o) {
      release();
      p = o.p; n = o.n; pool = std::move(o.pool); bytes = o.bytes;
      o.p = nullptr; o.n = 0;
    }
    return *this;
  }
  ~DBuf() { release(); }
  void alloc(size_t count) {
    release();
    if (!count) return;
    pool = current_pool();
    p = static_cast<T*>(pool ? pool->take(count * sizeof(T), bytes) : MemPool::device_malloc(count * sizeof(T)));
    n = count;
  }
  void release() {
    if (p) {
      if (pool) pool->give(p, bytes);
      else cudaFree(p);
    }
    pool.reset();
    p = nullptr; n = 0;
  }
  T* get() const { return p; }

 private:
  std::shared_ptr<MemPool> pool;   // where the block goes back to (null: cudaFree)
  size_t bytes = 0;                // the pool block's size
};

}  // namespace fsi
