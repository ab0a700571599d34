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
#include <mutex>
#include <unordered_map>
#include <vector>

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
        auto best = idle_.end();
        for (auto b = idle_.begin(); b != idle_.end(); ++b)
            if (b->dev == dev && b->size >= size && b->size <= 2 * size && (best == idle_.end() || b->size < best->size)) best = b;
        if (best != idle_.end()) {
            *p = best->p;
            live_[best->p] = *best;
            idle_.erase(best);
            return 0;
        }
        const int e = allocate(dev, size, p);
        if (e == 0) live_[*p] = Block{*p, size, dev};
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
        size_t bytes = 0, blocks = 0;
        for (const Block &b : idle_)
            if (b.dev == dev) {
                bytes += b.size;
                ++blocks;
            }
        for (auto b = idle_.begin(); b != idle_.end() && (bytes > kIdleBytes || blocks > kIdleBlocks);) {
            if (b->dev != dev) {
                ++b;
                continue;
            }
            bytes -= b->size;
            --blocks;
            Ops::release(b->p, b->dev);
            b = idle_.erase(b);
        }
    }

    // Frees the idle blocks of device dev (dev < 0: of every device).
    void release(int dev)
    {
        std::lock_guard<std::mutex> g(mu_);
        release_idle(dev);
    }

private:
    struct Block {
        void *p;
        size_t size;
        int dev;
    };
    std::mutex mu_;
    std::vector<Block> idle_;  // oldest first
    std::unordered_map<void *, Block> live_;

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
            if (dev >= 0 && b->dev != dev) {
                ++b;
                continue;
            }
            Ops::release(b->p, b->dev);
            b = idle_.erase(b);
            any = true;
        }
        return any;
    }
};

}  // namespace gbmc
