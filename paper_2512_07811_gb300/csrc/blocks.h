// Device blocks that a context has freed, kept for its next allocations of the
// same size class.  Plain C++: the driver is reached through BlockDevice.
//
// All work of a context runs on its one stream, so a block may be handed out
// again at once: its new user's kernels come after its last user's.  It saves
// two driver calls per buffer; a solve's six load-case threads queue on the
// driver's lock (about 30 buffers per rounded core; 16^3 elastic solve 140 / 110 ms).
//
// Bounded: a block above 64 MiB, or beyond 512 MiB in all contexts of the process
// together, goes back to the driver.  When an allocation fails, the cached blocks
// of every context on the device are given back first, and the size itself is
// asked for instead of its class.  Size classes: eight per power of two up to 1
// MiB, 32 above (at most 3 % more than asked for), none above 64 MiB.
//
// Stream capture: an allocation becomes a node of the graph and never enters the
// cache, none is taken from it, and a block from before the capture that is freed
// inside it is held until the context ends, since every replay of the graph
// may still read or write it.
//
// Locked, as several host threads may use one context, and a failed allocation
// reaches the caches of others.
#pragma once

#include <stddef.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <unordered_map>
#include <vector>

struct BlockDevice {
  virtual ~BlockDevice() {}
  virtual int id() = 0;                            // blocks of contexts with the same id share one memory
  virtual bool alloc(void** p, size_t bytes) = 0;  // on the context's stream
  virtual void release(void* p) = 0;               // on the context's stream
  virtual bool capturing() = 0;
  virtual void settle() = 0;  // returns once released blocks can serve other streams
};

class BlockCache {
 public:
  static constexpr size_t kMaxBlock = (size_t)64 << 20, kMaxTotal = (size_t)512 << 20;

  explicit BlockCache(BlockDevice* dev) : dev_(dev) {
    std::lock_guard<std::mutex> lk(registry_mu());
    registry().push_back(this);
  }
  ~BlockCache() { leave(); }
  BlockCache(const BlockCache&) = delete;
  BlockCache& operator=(const BlockCache&) = delete;

  static size_t size_class(size_t bytes) {
    if (bytes <= 512) return 512;
    if (bytes > kMaxBlock) return bytes;
    const int top = bytes > ((size_t)1 << 20) ? 6 : 4;  // bits of the leading part
    int sh = 0;
    while ((bytes - 1) >> (sh + top)) ++sh;
    return (((bytes - 1) >> sh) + 1) << sh;
  }

  bool alloc(void** p, size_t bytes) {
    if (dev_->capturing()) return dev_->alloc(p, bytes);
    const size_t cls = size_class(bytes);
    {
      std::lock_guard<std::mutex> lk(mu_);
      auto it = free_.find(cls);
      if (it != free_.end() && !it->second.empty()) {
        *p = it->second.back();
        it->second.pop_back();
        add_cached(-(ptrdiff_t)cls);
        return true;
      }
    }
    if (dev_->alloc(p, cls)) {
      if (cls <= kMaxBlock) {
        std::lock_guard<std::mutex> lk(mu_);
        size_of_[*p] = cls;
      }
      return true;
    }
    release_all();
    return dev_->alloc(p, bytes);  // (not of a class's size: not cached when freed)
  }

  void free(void* p) {
    const bool capturing = dev_->capturing();
    {
      std::lock_guard<std::mutex> lk(mu_);
      auto it = size_of_.find(p);
      if (it != size_of_.end()) {
        const size_t cls = it->second;
        if (capturing) {
          size_of_.erase(it);
          held_.push_back(p);
          return;
        }
        if (add_cached((ptrdiff_t)cls)) {
          free_[cls].push_back(p);
          return;
        }
        size_of_.erase(it);
      }
    }
    dev_->release(p);
  }

  // every cached block back to the driver (not while the stream is captured); whether there was one
  bool release() {
    if (dev_->capturing()) return false;
    std::lock_guard<std::mutex> lk(mu_);
    const bool any = !free_.empty();
    for (auto& l : free_)
      for (void* p : l.second) {
        size_of_.erase(p);
        add_cached(-(ptrdiff_t)l.first);
        dev_->release(p);
      }
    free_.clear();
    return any;
  }
  // at the end of the context, before its stream goes: also the blocks that a capture held
  void finish() {
    leave();
    release();
    std::lock_guard<std::mutex> lk(mu_);
    for (void* p : held_) dev_->release(p);
    held_.clear();
  }

 private:
  void release_all() {
    std::lock_guard<std::mutex> lk(registry_mu());
    for (BlockCache* b : registry())
      if (b->dev_->id() == dev_->id() && b->release() && b != this) b->dev_->settle();
  }
  // no other context's failed allocation comes here any more
  void leave() {
    std::lock_guard<std::mutex> lk(registry_mu());
    auto& r = registry();
    r.erase(std::remove(r.begin(), r.end(), this), r.end());
  }
  // false where the bound does not allow it (one counter for all contexts, no lock: every
  // allocation and release of a solve's threads comes here)
  static bool add_cached(ptrdiff_t n) {
    static std::atomic<ptrdiff_t>& total = *new std::atomic<ptrdiff_t>(0);
    const ptrdiff_t now = total.fetch_add(n) + n;
    if (n > 0 && now > (ptrdiff_t)kMaxTotal) {
      total.fetch_sub(n);
      return false;
    }
    return true;
  }
  static std::mutex& registry_mu() {
    static std::mutex& m = *new std::mutex;  // (contexts may end after static objects do)
    return m;
  }
  static std::vector<BlockCache*>& registry() {
    static std::vector<BlockCache*>& r = *new std::vector<BlockCache*>;
    return r;
  }

  BlockDevice* dev_;
  std::mutex mu_;
  std::unordered_map<void*, size_t> size_of_;     // blocks of a class's size, in use or cached
  std::map<size_t, std::vector<void*>> free_;     // by size class
  std::vector<void*> held_;
};
