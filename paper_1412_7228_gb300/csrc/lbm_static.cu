// lbm_static.cu -- lbm_field_pressure_jump_static: the Laplace-law sums of
// lbm_batch_measure over a density field the caller already holds in device
// memory, with no device allocation of any kind.
//
// Who needs it: code that cannot call cudaMalloc -- for example a caller whose
// device memory is entirely owned by another allocator (a framework's caching
// allocator or a fixed arena reserved at start-up, where a fresh cudaMalloc
// fails or breaks the memory budget), or a latency-critical loop that must not
// pay for an allocation call that can synchronise the whole device.  Those
// callers pass the input field and a host output array and nothing else.
//
// Scratch: the per-block partial sums live in g_scratch, a file-scope
// __device__ array.  Every GPU that loads this library holds it (about 128 KiB)
// until the process exits.  Host code cannot use the symbol itself as a device
// address, so the first call on each device looks its address up with
// cudaGetSymbolAddress (with that device current) and caches it; make that
// first call before any stream capture begins.  Every call copies its eight
// totals to host memory and synchronises its stream before it returns.  All
// calls share the array and it keeps the previous call's contents: each
// block writes every slot it later reads, and each call clears the ticket
// first (so calls that raced cannot spoil a later one), but two calls whose
// kernels overlap on the GPU (different streams or host threads) race on it.
//
// The field must be device memory of the current device: the call checks
// this (cudaPointerGetAttributes) and rejects anything else with
// LBM_EINVAL, as it rejects an equation of state that lbm_set_params would
// reject, before any GPU work.
#include <cmath>
#include <cstring>
#include <mutex>

#include "lbm_eos_host.h"
#include "lbm_internal.cuh"
#include "lbm_reduce.cuh"

namespace lbm {
namespace {

constexpr int kSlots = 8;
constexpr int kStaticBlocks = 8 * 152;   // resident blocks of a 152-SM GB300: partial sums of the largest grid
constexpr int kScratchRows = 2048;

// partial sums of the blocks, then the 8 totals, then the ticket of the last
// block
static __device__ __align__(256) double g_scratch[kScratchRows * kSlots + kSlots + 1];
static_assert(kStaticBlocks <= kScratchRows, "one row of partial sums per block");

constexpr int kMaxDevices = 64;
std::mutex g_mu;
double* g_ptr[kMaxDevices] = {};

// The Laplace sums of a field (LaplaceSums) in one launch, bound by the FP64
// pipe (17.5 instructions per node; 4096^2: 1970 -> 689 us per call, 617 on the
// device; the former second launch was 168).  EXACT: see LawFp64.
template <bool EXACT>
__global__ void __launch_bounds__(kLapThreads)
    k_field_sums(const double* __restrict__ rho, int nx, int ny, Phys<double> P, Discs D, int rpt,
                 double* __restrict__ partials, unsigned* ticket, double* __restrict__ out) {
    __shared__ AxisTable A;
    LaplaceSums<EXACT> L;
    laplace_tiles(L, LawFp64(P, false), D, nx, ny, rpt, A,
                  [&](int x, int y) { return rho[static_cast<long long>(y) * nx + x]; });
    double total;
    if (grid_sum8<kLapThreads>(L.v, -1, 0.0, partials, ticket, &total)) out[threadIdx.x] = total;
}

// Address of g_scratch on the current device, looked up once per device.
cudaError_t scratch_on_current_device(double** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess) return e;
        g_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_ptr[dev];
    return cudaSuccess;
}

// d_rho is device (or managed) memory whose device is the current one.
bool on_current_device(const void* p) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();   // the query's own error, not a pending one of the caller
        return false;
    }
    return (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == dev;
}

}  // namespace
}  // namespace lbm

extern "C" int lbm_field_pressure_jump_static(const double* d_rho, int nx, int ny, const lbm_eos* eos, double cx,
                                              double cy, double r_in, double r_out, double* out, void* stream) {
    using namespace lbm;
    if (!d_rho || !out || nx < 1 || ny < 1 || !(r_in >= 0) || !(r_out >= 0)) return LBM_EINVAL;
    if (!std::isfinite(cx) || !std::isfinite(cy) || !std::isfinite(r_in) || !std::isfinite(r_out)) return LBM_EINVAL;
    if (!eos_valid_at(eos)) return LBM_EINVAL;   // the laws and temperatures lbm_set_params accepts
    const long long N = static_cast<long long>(nx) * ny;
    if (N > LBM_STATIC_MAX_NODES) return LBM_EINVAL;   // the static scratch holds partials for at most this many nodes
    if (!on_current_device(d_rho)) return LBM_EINVAL;
    double* scratch = nullptr;
    if (scratch_on_current_device(&scratch) != cudaSuccess) return LBM_ECUDA;

    Phys<double> P;
    std::memset(&P, 0, sizeof P);
    fill_eos(P, *eos);

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Discs D = make_discs(nx, ny, cx, cy, r_in, r_out);
    int rpt = tile_rpt(nx, ny);
    const long long tiles = tile_count(nx, ny, rpt);
    const int blocks = static_cast<int>(tiles < kStaticBlocks ? tiles : kStaticBlocks);
    double* partials = scratch;
    double* totals = scratch + kScratchRows * kSlots;
    unsigned* ticket = reinterpret_cast<unsigned*>(totals + kSlots);
    // cudaLaunchKernel returns this launch's own error (never an earlier one)
    void* args[] = {&d_rho, &nx, &ny, &P, &D, &rpt, &partials, &ticket, &totals};
    double s[kSlots];
    for (const void* kernel : {reinterpret_cast<const void*>(&k_field_sums<false>),
                               reinterpret_cast<const void*>(&k_field_sums<true>)}) {
        if (cudaMemsetAsync(ticket, 0, sizeof *ticket, st) != cudaSuccess ||
            cudaLaunchKernel(kernel, dim3(blocks), dim3(kLapThreads), args, 0, st) != cudaSuccess ||
            cudaMemcpyAsync(s, totals, sizeof s, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return LBM_ECUDA;
        if (!on_the_pole(s)) break;
    }

    const double p_in = s[3] > 0 ? s[1] / s[3] : NAN, rho_in = s[3] > 0 ? s[2] / s[3] : NAN;
    const double p_out = s[6] > 0 ? s[4] / s[6] : NAN, rho_out = s[6] > 0 ? s[5] / s[6] : NAN;
    const double ex = s[0] - rho_out * static_cast<double>(N);
    const double R_eq = std::sqrt((ex > 0 ? ex : 0.0) / (M_PI * (rho_in - rho_out)));
    const double vals[LBM_MEASURE_N] = {p_in, p_out, rho_in, rho_out, R_eq, s[0], s[3], s[6]};
    std::memcpy(out, vals, sizeof vals);
    return LBM_OK;
}
