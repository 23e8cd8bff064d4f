// lbm_pinned.cu -- pinned host memory, mapped for the devices, of the contexts
// and networks.  It comes in slabs: of 256 blocks for what each context keeps
// (64 KB), and of 8 for the networks and for the stage of small pageable
// read-backs (half a megabyte), so that making a context costs no
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
    const void* context() {
        static const auto current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
        CUcontext c = nullptr;
        if (current && current(&c) == CUDA_SUCCESS && !c) {   // the runtime makes its own current on first use
            cudaFree(nullptr);
            current(&c);
        }
        return c;
    }
    unsigned long long id(void* p) {
        static const auto get =
            driver_function<CUresult (*)(void*, CUpointer_attribute, CUdeviceptr)>("cuPointerGetAttribute");
        unsigned long long v = 0;
        return get && get(&v, CU_POINTER_ATTRIBUTE_BUFFER_ID, reinterpret_cast<CUdeviceptr>(p)) == CUDA_SUCCESS ? v : 0;
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

HostMemory host_memory(const void* p) {
    static const auto get =
        driver_function<CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr)>("cuPointerGetAttributes");
    HostMemory m = {};
    unsigned type = 0, managed = 0;   // type 0: unknown
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                  CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* to[] = {&type, &managed, &m.device, &m.range.at, &m.range.bytes};
    if (!get || get(5, what, to, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS) {
        m.known = true;   // left to the copies
        return m;
    }
    m.known = type != 0 || managed != 0;
    m.pinned = type == CU_MEMORYTYPE_HOST && !managed && m.device;
    return m;
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
