// lbm_pinned.cu -- pinned host memory, mapped for the devices, of the contexts
// and networks.  Allocating and freeing it takes the driver about 100 and 180 us,
// three times what making a small context takes otherwise, so the first
// owner allocates a slab of kBlocks blocks of one size, which serves up to
// that many owners at a time and is given back at exit; further owners, and
// larger requests, go to the driver.  A block's owner has waited for its
// stream before it lets go.
#include <mutex>

#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kBlocks = 8;   // half a megabyte

struct Pool {
    std::mutex mu;
    char* slab = nullptr;
    bool used[kBlocks] = {};
    ~Pool() {
        if (slab) cudaFreeHost(slab);
    }
    // a free block of the slab, or NULL
    void* take() {
        std::lock_guard<std::mutex> lock(mu);
        if (!slab) slab = static_cast<char*>(allocate(kBlocks * kPinnedBlock));
        for (int k = 0; slab && k < kBlocks; ++k)
            if (!used[k]) {
                used[k] = true;
                return slab + k * kPinnedBlock;
            }
        return nullptr;
    }
    // whether p was a block of the slab, now free again
    bool put(void* p) {
        std::lock_guard<std::mutex> lock(mu);
        for (int k = 0; slab && k < kBlocks; ++k)
            if (p == slab + k * kPinnedBlock) {
                used[k] = false;
                return true;
            }
        return false;
    }
    static void* allocate(size_t bytes) {
        void* v = nullptr;
        if (cudaHostAlloc(&v, bytes, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) return v;
        cudaGetLastError();
        return nullptr;
    }
};
Pool& pool() {
    static Pool p;
    return p;
}

}  // namespace

bool pointer_attribute(CUpointer_attribute what, const void* p, void* out) {
    typedef CUresult (*Get)(void*, CUpointer_attribute, CUdeviceptr);
    static const Get get = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &fn, 12000, cudaEnableDefault, &q) ==
                            cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<Get>(fn) : nullptr;
    }();
    return get && get(out, what, reinterpret_cast<CUdeviceptr>(p)) == CUDA_SUCCESS;
}

void* pinned_get(size_t bytes) {
    if (bytes <= kPinnedBlock)
        if (void* p = pool().take()) return p;
    return Pool::allocate(bytes);
}

void pinned_put(void* p) {
    if (p && !pool().put(p)) cudaFreeHost(p);
}

}  // namespace lbm
