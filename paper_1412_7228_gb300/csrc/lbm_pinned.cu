// lbm_pinned.cu -- pinned host memory, mapped for the devices, of the contexts
// and networks.  Allocating and freeing it takes the driver about 100 and 180 us,
// three times what making a small context takes otherwise, so the first
// owner allocates a slab of kBlocks blocks of one size, which serves up to
// that many owners at a time and is given back at exit; further owners, and
// larger requests, go to the driver.  A block's owner has waited for its
// stream before it lets go.  The bookkeeping is lbm_pinned_pool.h's.
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kBlocks = 8;   // half a megabyte

// A function of the driver, which the library does not link.
template <class F> F driver_function(const char* name) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPointByVersion(name, &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    return ok ? reinterpret_cast<F>(fn) : nullptr;
}

struct CudaDriver {
    void* allocate(size_t bytes) {
        void* v = nullptr;
        if (cudaHostAlloc(&v, bytes, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) return v;
        cudaGetLastError();
        return nullptr;
    }
    void release(void* p) { cudaFreeHost(p); }
    unsigned long long context() {
        static const auto current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
        static const auto id_of = driver_function<CUresult (*)(CUcontext, unsigned long long*)>("cuCtxGetId");
        CUcontext c = nullptr;
        unsigned long long id = 0;
        if (!current || !id_of) return 0;
        if (current(&c) == CUDA_SUCCESS && !c) {   // the runtime makes its own current on first use
            cudaFree(nullptr);
            current(&c);
        }
        return c && id_of(c, &id) == CUDA_SUCCESS ? id : 0;
    }
    unsigned long long id(void* p) {
        unsigned long long v = 0;
        return pointer_attribute(CU_POINTER_ATTRIBUTE_BUFFER_ID, p, &v) ? v : 0;
    }
};
PinnedPool<CudaDriver>& pool() {
    static PinnedPool<CudaDriver> p(kPinnedBlock, kBlocks);
    return p;
}

}  // namespace

bool pointer_attribute(CUpointer_attribute what, const void* p, void* out) {
    static const auto get = driver_function<CUresult (*)(void*, CUpointer_attribute, CUdeviceptr)>("cuPointerGetAttribute");
    return get && get(out, what, reinterpret_cast<CUdeviceptr>(p)) == CUDA_SUCCESS;
}

Pinned pinned_get(size_t bytes) { return pool().get(bytes); }

void pinned_put(const Pinned& b) { pool().put(b); }

}  // namespace lbm
