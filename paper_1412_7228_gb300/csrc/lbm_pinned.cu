// lbm_pinned.cu -- pinned host memory, mapped for the devices, of the contexts
// and networks.  Allocating and freeing it takes the driver about 100 and 180 us,
// three times what making a small context takes otherwise, so blocks of
// one size are kept for the next owner: at most kKept of them, given back at
// exit.  A block's former owner has waited for its stream before it lets go.
#include <mutex>

#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kKept = 8;   // half a megabyte

struct Pool {
    std::mutex mu;
    void* block[kKept] = {};
    int n = 0;
    ~Pool() {
        for (int k = 0; k < n; ++k) cudaFreeHost(block[k]);
    }
};
Pool& pool() {
    static Pool p;
    return p;
}

}  // namespace

void* pinned_get(size_t bytes) {
    if (bytes <= kPinnedBlock) {
        Pool& p = pool();
        std::lock_guard<std::mutex> lock(p.mu);
        if (p.n > 0) return p.block[--p.n];
    }
    void* v = nullptr;
    const size_t size = bytes <= kPinnedBlock ? kPinnedBlock : bytes;
    if (cudaHostAlloc(&v, size, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return v;
}

void pinned_put(void* v, size_t bytes) {
    if (!v) return;
    if (bytes <= kPinnedBlock) {
        Pool& p = pool();
        std::lock_guard<std::mutex> lock(p.mu);
        if (p.n < kKept) {
            p.block[p.n++] = v;
            return;
        }
    }
    cudaFreeHost(v);
}

}  // namespace lbm
