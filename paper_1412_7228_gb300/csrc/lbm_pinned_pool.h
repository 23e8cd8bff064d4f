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
#include <cstddef>
#include <mutex>
#include <vector>

namespace lbm {

struct Pinned {
    void* p = nullptr;
    unsigned long long slab = 0;   // 0: straight from the driver
};

// Driver: void* allocate(size_t); void release(void*); const void* context(),
// the current context (one made later may have the handle of a lost one), and
// unsigned long long id(void*), the process-wide id of the live allocation at
// an address (0: none).
//
// A context whose slabs are all taken gets another, and one that becomes empty
// is given back unless it is the context's only empty one: the pinned memory
// follows the owners that are alive, and a slab's cost is spread over them.
template <class Driver> class PinnedPool {
public:
    PinnedPool(size_t block, int blocks) : block_(block), blocks_(blocks) {}
    ~PinnedPool() {
        for (Slab& s : slabs_)
            if (alive(s)) driver_.release(s.base);
    }
    // a block, or where there is no slab for it memory of its own
    Pinned get() {
        Pinned b = take();
        if (!b.p) b.p = driver_.allocate(block_);
        return b;
    }
    // whether b was one of this pool's slabs' blocks, now free again
    bool put(const Pinned& b) {
        std::lock_guard<std::mutex> lock(mu_);
        const auto from = std::find_if(slabs_.begin(), slabs_.end(), [&](const Slab& s) { return s.id == b.slab; });
        if (from == slabs_.end()) return false;
        from->used[static_cast<size_t>(static_cast<char*>(b.p) - from->base) / block_] = 0;
        if (--from->taken) return true;
        for (const Slab& s : slabs_)
            if (s.id != from->id && s.context == from->context && !s.taken) {
                if (alive(*from)) driver_.release(from->base);
                slabs_.erase(from);
                break;
            }
        return true;
    }
    Driver& driver() { return driver_; }

private:
    struct Slab {
        char* base;
        unsigned long long id;
        const void* context;
        std::vector<char> used;
        int taken;
    };
    bool alive(const Slab& s) { return driver_.id(s.base) == s.id; }
    // a free block of the current context's slabs, or none
    Pinned take() {
        std::lock_guard<std::mutex> lock(mu_);
        const void* const context = driver_.context();
        Slab* from = nullptr;
        for (size_t k = 0; k < slabs_.size() && !from;) {
            Slab& s = slabs_[k];
            if (s.context != context || s.taken == blocks_) ++k;
            else if (alive(s)) from = &s;
            else slabs_.erase(slabs_.begin() + static_cast<std::ptrdiff_t>(k));   // its context is gone
        }
        if (!from) {
            void* const base = driver_.allocate(block_ * blocks_);
            if (!base) return {};
            const unsigned long long id = driver_.id(base);
            if (!id) {   // without one it could not be told from another
                driver_.release(base);
                return {};
            }
            slabs_.push_back({static_cast<char*>(base), id, context, std::vector<char>(blocks_, 0), 0});
            from = &slabs_.back();
        }
        const size_t k = std::find(from->used.begin(), from->used.end(), 0) - from->used.begin();
        from->used[k] = 1;
        ++from->taken;
        Pinned b;
        b.p = from->base + k * block_;
        b.slab = from->id;
        return b;
    }

    const size_t block_;
    const int blocks_;
    std::mutex mu_;
    std::vector<Slab> slabs_;
    Driver driver_;
};

}  // namespace lbm
