// lbm_pinned.cu -- pinned host memory, mapped for the devices, of the contexts
// and networks.  It comes in slabs: of 256 blocks for what each context keeps
// (64 KB), and of 8 for the networks and for the stage that a read-back borrows
// while it lasts (half a megabyte), so that making a context costs no
// allocation by the driver however many are open (64 of 64^2 at once: 23.3 us to
// make and 1.1 to close each; with an allocation of its own for each beyond the
// eighth 30.0 and 6.7).  Larger requests go to the driver.  A block's owner has waited
// for its stream before it lets go.  The bookkeeping is lbm_pinned_pool.h's.
#include "lbm_internal.cuh"

namespace lbm {
namespace {

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
PinnedPool<CudaDriver>& small_pool() {
    static PinnedPool<CudaDriver> p(kPinnedSmall, 256);
    return p;
}
PinnedPool<CudaDriver>& pool() {
    static PinnedPool<CudaDriver> p(kPinnedBlock, 8);
    return p;
}

}  // namespace

bool pointer_attribute(CUpointer_attribute what, const void* p, void* out) {
    static const auto get = driver_function<CUresult (*)(void*, CUpointer_attribute, CUdeviceptr)>("cuPointerGetAttribute");
    return get && get(out, what, reinterpret_cast<CUdeviceptr>(p)) == CUDA_SUCCESS;
}

Pinned pinned_get(size_t bytes) {
    if (bytes <= kPinnedSmall) return small_pool().get();
    if (bytes <= kPinnedBlock) return pool().get();
    Pinned b;
    b.p = CudaDriver().allocate(bytes);
    return b;
}

void pinned_put(const Pinned& b) {
    if (b.slab) small_pool().put(b) || pool().put(b);
    else if (b.p) CudaDriver().release(b.p);
}

}  // namespace lbm
