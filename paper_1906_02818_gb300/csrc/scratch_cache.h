// Device allocations of the library, behind the calls that make them (host
// code without CUDA headers, so that it is tested with an allocator that
// fails on request).
//
// Scratch comes from a cache of freed blocks (per device; sizes rounded up to
// 256 bytes; a request takes the smallest free block of at least its size and
// at most twice it), so that repeated calls of the same shape pay neither
// cudaMalloc nor cudaFree (which also synchronises the device).  A block goes
// back to the cache only when no launch can still use it (its owner has
// synchronised).  What lies idle is bounded: past kIdleBytes or kIdleBlocks of
// a device its oldest blocks are freed.  8 GiB are 3 % of the card and hold the
// largest set of buffers that a call of the workloads in use asks for again
// and again (4.3 GB: correlation sensitivities of 512 assets, 2^20 paths).
// Where the device is short of memory, the idle blocks are handed back and the
// request is tried once more, whether or not it is for the cache.
#pragma once

#include <cstddef>
#include <iterator>
#include <list>
#include <map>
#include <mutex>
#include <unordered_map>
#include <utility>

namespace gbmc {

// Ops::allocate(p, n): n bytes on the current device; 0 or an error code, which
// leaves no error pending; Ops::kNoMemory where memory is short.
// Ops::release(p, dev): frees a block of device dev.
template <class Ops>
class ScratchCache {
public:
    static constexpr size_t kIdleBytes = size_t(8) << 30, kIdleBlocks = 1024;

    // A block of at least n bytes on device dev (the current one).
    int take(int dev, size_t n, void **p)
    {
        const size_t size = n <= 256 ? 256 : (n + 255) & ~static_cast<size_t>(255);
        std::lock_guard<std::mutex> g(mu_);
        const auto best = by_size_.lower_bound({dev, size});
        if (best != by_size_.end() && best->first.first == dev && best->first.second <= 2 * size) {
            const Block b = *best->second;
            drop(best->second);
            live_[b.p] = b;
            *p = b.p;
            return 0;
        }
        const int e = allocate(dev, size, p);
        if (e == 0) live_[*p] = Block{*p, size, dev, {}};
        return e;
    }

    // The same past the cache: the caller frees it.
    int take_uncached(int dev, size_t n, void **p)
    {
        std::lock_guard<std::mutex> g(mu_);
        return allocate(dev, n, p);
    }

    void give(void *p)
    {
        if (!p) return;
        std::lock_guard<std::mutex> g(mu_);
        const auto it = live_.find(p);
        if (it == live_.end()) return;
        const Block given = it->second;
        const int dev = given.dev;
        live_.erase(it);
        if (given.size > kIdleBytes) {  // would only drive the others out
            Ops::release(given.p, dev);
            return;
        }
        idle_.push_back(given);
        idle_.back().at = by_size_.insert({{dev, given.size}, std::prev(idle_.end())});
        Total &t = total_[dev];
        t.bytes += given.size;
        ++t.blocks;
        for (auto b = idle_.begin(); t.bytes > kIdleBytes || t.blocks > kIdleBlocks;) {
            const auto old = b++;
            if (old->dev != dev) continue;
            const Block gone = *old;
            drop(old);
            Ops::release(gone.p, dev);
        }
    }

    // Frees the idle blocks of device dev (dev < 0: of every device).
    void release(int dev)
    {
        std::lock_guard<std::mutex> g(mu_);
        release_idle(dev);
    }

private:
    struct Block;
    using Idle = std::list<Block>;  // oldest first
    using Index = std::multimap<std::pair<int, size_t>, typename Idle::iterator>;  // by device and size
    struct Block {
        void *p;
        size_t size;
        int dev;
        typename Index::iterator at;  // idle blocks: the entry of the index
    };
    struct Total {
        size_t bytes = 0, blocks = 0;
    };
    std::mutex mu_;
    Idle idle_;
    Index by_size_;
    std::map<int, Total> total_;  // idle, by device
    std::unordered_map<void *, Block> live_;

    void drop(typename Idle::iterator b)
    {
        Total &t = total_[b->dev];
        t.bytes -= b->size;
        --t.blocks;
        by_size_.erase(b->at);
        idle_.erase(b);
    }
    int allocate(int dev, size_t n, void **p)
    {
        int e = Ops::allocate(p, n);
        if (e == Ops::kNoMemory && release_idle(dev)) e = Ops::allocate(p, n);
        return e;
    }
    bool release_idle(int dev)
    {
        bool any = false;
        for (auto b = idle_.begin(); b != idle_.end();) {
            const auto old = b++;
            if (dev >= 0 && old->dev != dev) continue;
            const Block gone = *old;
            drop(old);
            Ops::release(gone.p, gone.dev);
            any = true;
        }
        return any;
    }
};

}  // namespace gbmc
