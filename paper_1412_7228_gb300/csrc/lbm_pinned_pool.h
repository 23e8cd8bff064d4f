// lbm_pinned_pool.h -- small blocks of pinned host memory cut from slabs
// (lbm_pinned.cu), over a Driver that allocates, so that the bookkeeping can be
// tested without a GPU.
//
// Pinned memory belongs to the CUDA context that it was allocated in and goes
// with it (cuCtxDestroy, cudaDeviceReset), so each context has its own
// slab, a slab is used again only while the driver still knows it by the id
// that it had when it was made, and a block is given back by that id: never
// into another slab that has come to lie at the same address.
#pragma once

#include <stddef.h>

#include <algorithm>
#include <mutex>
#include <vector>

namespace lbm {

struct Pinned {
    void* p = nullptr;
    unsigned long long slab = 0;   // 0: straight from the driver
};

// Driver: void* allocate(size_t); void release(void*); the process-wide ids
// unsigned long long context() of the current context and
// unsigned long long id(void*) of the live allocation at an address (0: none).
template <class Driver> class PinnedPool {
public:
    PinnedPool(size_t block, int blocks) : block_(block), blocks_(blocks) {}
    ~PinnedPool() {
        for (Slab& s : slabs_)
            if (alive(s)) driver_.release(s.base);
    }
    Pinned get(size_t bytes) {
        if (bytes <= block_) {
            const Pinned b = take();
            if (b.p) return b;
        }
        Pinned b;
        b.p = driver_.allocate(bytes);
        return b;
    }
    void put(const Pinned& b) {
        if (!b.p) return;
        if (!b.slab) {
            driver_.release(b.p);
            return;
        }
        std::lock_guard<std::mutex> lock(mu_);
        for (Slab& s : slabs_)
            if (s.id == b.slab) s.used[static_cast<size_t>(static_cast<char*>(b.p) - s.base) / block_] = 0;
    }
    Driver& driver() { return driver_; }

private:
    struct Slab {
        char* base;
        unsigned long long id, context;
        std::vector<char> used;
    };
    bool alive(const Slab& s) { return driver_.id(s.base) == s.id; }
    // a free block of the current context's slab, or none
    Pinned take() {
        std::lock_guard<std::mutex> lock(mu_);
        slabs_.erase(std::remove_if(slabs_.begin(), slabs_.end(), [&](const Slab& s) { return !alive(s); }), slabs_.end());
        const unsigned long long context = driver_.context();
        Slab* mine = nullptr;
        for (Slab& s : slabs_)
            if (s.context == context) mine = &s;
        if (!mine) {
            void* const base = driver_.allocate(block_ * blocks_);
            if (!base) return {};
            const unsigned long long id = driver_.id(base);
            if (!id) {   // without one it could not be told from another
                driver_.release(base);
                return {};
            }
            slabs_.push_back({static_cast<char*>(base), id, context, std::vector<char>(blocks_, 0)});
            mine = &slabs_.back();
        }
        for (int k = 0; k < blocks_; ++k)
            if (!mine->used[k]) {
                mine->used[k] = 1;
                Pinned b;
                b.p = mine->base + k * block_;
                b.slab = mine->id;
                return b;
            }
        return {};
    }

    const size_t block_;
    const int blocks_;
    std::mutex mu_;
    std::vector<Slab> slabs_;
    Driver driver_;
};

}  // namespace lbm
