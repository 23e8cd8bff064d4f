// lbm_internal.cuh -- device data layout, per-instance descriptors and the
// PTX helpers (mbarrier, TMA) shared by the sm_103a kernels of liblbm.
//
// HBM layout of one instance in precision T (float: deviations from
// t_a rho_ref; double: same, rho_ref may be 0):
//   pop[k][a][Y][X],  k in {0,1} the two time levels, a = 0..8,
//   Y = y + GY (GY = 2 ghost rows above and below),
//   X = x + GX (GX = 32 bytes / sizeof(T) ghost columns on the left, so an
//   interior row starts on a 32-byte sector), row pitch a multiple of 32 B.
// The array holds post-collision populations at their source node ("pull"
// storage): the pre-collision f_a(x, t) is pop[a][x - e_a].  Ghost cells
// hold periodic images, written by the step kernel for border nodes, so a
// tile's halo is one rectangular TMA box with no wrap logic.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lbm.h"
#include "lbm_host_rules.h"
#include "lbm_pinned_pool.h"

namespace lbm {

constexpr int GY = 2;          // ghost rows per side
constexpr int kMaxSched = 5;   // CTA schedules known to lbm_set_schedule (3: multi-step persistent, 4: cluster)

template <typename T> struct Prec;
template <> struct Prec<float> { static constexpr int GX = 8; static constexpr int HX = 4; };
template <> struct Prec<double> { static constexpr int GX = 4; static constexpr int HX = 2; };

// Lattice velocity components e_a.
__host__ __device__ constexpr int cx(int a) {
    return (a == 1 || a == 5 || a == 8) ? 1 : ((a == 3 || a == 6 || a == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cy(int a) {
    return (a == 2 || a == 5 || a == 6) ? 1 : ((a == 4 || a == 7 || a == 8) ? -1 : 0);
}

// Status bits of an instance (sticky until cleared or re-initialised).
constexpr int ST_UNSTABLE = 1;
constexpr int ST_TIMEOUT = 2;

// Constants of one precision's node only, formed once on the host: FP32
// (collide in lbm_step_kernels.cuh) and FP64 (collide64).  Apart, they leave
// Inst, and so the memory that a context asks for, as small as it was before
// FP64 had its own.
template <typename T> struct NodeConsts;
template <> struct NodeConsts<float> {
    float nhs[9];                // -(1 - s/2)
};
template <> struct NodeConsts<double> {
    double cF, hF;               // -(G/12) (1 - A), -(G/12) A/2
    double k1[3], k1r, k1q;      // e*: f_0, axis sum, diagonal sum; rho|v|^2; tr Q's sum
    double k2[2], k2r, k2q;      // eps*: f_0, axis sum (diagonal sum: 1); likewise
    double k4[2], k6[2];         // q_x*, q_y*: axis and diagonal fluxes
    double k7q, k8q;             // p_xx*, p_xy*: the sums of Q_xx - Q_yy and Q_xy
};

// Physics parameters in the kernel's precision.
template <typename T> struct Phys : NodeConsts<T> {
    int eos;            // LBM_EOS_*
    unsigned flags;     // LBM_FLAG_*
    T K, a, b, b4, RT, aalpha;   // EOS; b4 = b/4 (CS), aalpha = a alpha(T) (PR)
    T A, kappa, G, two_over_G;   // Eq. 9, Eq. 23, Eq. 10
    T hs[9];            // 1 - s/2, the forcing weight of Eq. 5 (s: Lambda)
    T ns[9];            // -s
    T h2s7;             // 2 hs[7] (exact)
    T h6s1, nh6s2;      // 6 hs[1], -6 hs[2]: the forcing weights of S[1] = 6 v.F, S[2] = -6 v.F
    T c1, c2;           // C[1] = c1 tr Q, C[2] = c2 tr Q (Eq. 26)
    T rho_ref;          // deviation reference
    int interact;       // 0 when G == 0: no psi, F = Q = 0
    // density-dependent shear viscosity: nu(rho) linear between (rho_g, nu_g)
    // and (rho_l, nu_l), clamped; s_7 = s_8 = 1 / (3 nu + 1/2)
    int var_visc;
    T nu_g, dnu, visc_rho_g, visc_inv_drho;
};

// One lattice, as the kernels see it in global memory.  Its TMA tensor maps
// are not here: they travel in the kernel argument blocks below.
struct alignas(128) Inst {
    void* pop[2];
    int* status;
    int nx, ny, pitch, nyp;  // pitch, nyp in elements
    long long plane;         // pitch * nyp
    Phys<float> pf;
    Phys<double> pd;
    int prec;                // LBM_FP32 / LBM_FP64
    int pad_[3];
};

// Everything a single-lattice step needs, passed by value as a
// __grid_constant__ kernel argument: the tensor maps and constants then live
// in the parameter bank, and tile coordinates come from blockIdx.
template <typename T> struct StepArgs {   // CUtensorMap members give it their alignment
    CUtensorMap tmap[2];
    Phys<T> P;
    void* pop[2];
    int* status;
    long long plane;
    int nx, ny, pitch, tiles_x;
};

// What a batched launch needs, passed by value as a __grid_constant__
// kernel argument as well: for up to kBatchLaunchMax instances their tensor
// maps (in parameter space a map needs neither a load of its own nor a
// tensormap proxy fence, which a map in global memory needs before every
// first use in a CTA) and tile counts; in FP32 also their array addresses,
// sizes and constants, so that the FP32 step reads nothing but populations
// from global memory (FP64, bound by its FP64 pipe, reads those from the
// instance descriptors: 64 FP64 constant sets would not fit the 32 KB
// argument space).  Slot k's tiles are first[k] .. first[k+1]-1, row-major
// over tiles_x[k] columns; with a tile table (the interleaved schedule)
// entry t gives (slot << 24 | x0, y0) instead.  A batch with more instances is
// stepped by several launches.
constexpr int kBatchLaunchMax = 64;
struct SlotLattice {                     // the fields of Inst the step uses
    void* pop[2];
    int* status;
    long long plane;
    int nx, ny, pitch, pad_;
};
template <typename T> struct BatchPhys {};
template <> struct BatchPhys<float> {
    Phys<float> P[kBatchLaunchMax];
};
template <typename T> struct BatchArgs {
    CUtensorMap tmap[kBatchLaunchMax];   // maps of the source time level of slot k
    const int2* tiles;                   // tile table, or nullptr: tiles in slot order
    int first[kBatchLaunchMax + 1];      // first tile of slot k; first[n] = tiles of the launch
    int tiles_x[kBatchLaunchMax];        // tile columns of slot k
    unsigned div_m[kBatchLaunchMax];     // division by tiles_x[k]: see tile_row()
    int div_s[kBatchLaunchMax];
    int inst[kBatchLaunchMax];           // slot k -> index into the Inst array
    int n;                               // slots in use, 1..kBatchLaunchMax
    SlotLattice lat[kBatchLaunchMax];    // read by FP32 launches
    BatchPhys<T> phys;                   // FP32 only
};

// What a multi-step persistent launch needs (schedule 3): for up to
// kRunMax instances the tensor maps of both time levels, tile counts, array
// addresses and sizes, FP32 constants, and the launch's work counter and the
// per-tile step counters in global memory.  Work item w is step w / ntiles
// of tile w % ntiles (tiles in slot order, row-major within an instance); a
// CTA takes items in that order and starts step s of a tile once every tile
// within two nodes of it (periodic within the instance: its 3 x 3 tile
// neighbourhood, and the tile beyond a last tile row or column one node
// wide) has finished step s - 1.
constexpr int kRunMax = 32;
template <typename T> struct RunPhys {};
template <> struct RunPhys<float> {
    Phys<float> P[kRunMax];
};
template <typename T> struct RunArgs {
    CUtensorMap tmap[2][kRunMax];        // [time level][slot]
    int first[kRunMax + 1];              // first tile of slot k; first[n] = ntiles
    int tiles_x[kRunMax];                // tile columns of slot k
    int inst[kRunMax];                   // slot k -> index into the Inst array
    int n;                               // slots in use, 1..kRunMax
    int ntiles;                          // tiles of all slots
    int nsteps;                          // steps this launch performs
    int parity0;                         // time level the first step reads
    int* done;                           // per tile: steps it has completed in this launch
    unsigned long long* counter;         // next work item
    int* abort_flag;                     // set when a bounded wait gave up: every CTA stops
    SlotLattice lat[kRunMax];            // read by FP32 launches
    RunPhys<T> phys;                     // FP32 only
};

// kernel parameters are limited to 32,764 bytes
static_assert(sizeof(BatchArgs<float>) <= 32764 && sizeof(BatchArgs<double>) <= 32764, "argument block too large");
static_assert(sizeof(RunArgs<float>) <= 32764 && sizeof(RunArgs<double>) <= 32764, "argument block too large");

// floor(r / d) for 0 <= r < 2^31 and d >= 1 as one 64-bit multiply and a
// shift (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994): with l = ceil(log2 d), m = ceil(2^(31+l) / d) and
// s = 31 + l, m d - 2^s lies in [0, d - 1] and d <= 2^l, so
// r m / 2^s = r / d + e with 0 <= e < 1/d, which cannot reach the next
// integer; m < 2^32.  The host computes (m, s) per instance and checks the
// result for every tile it launches.
__host__ __device__ __forceinline__ int tile_row(int r, unsigned m, int s) {
    return static_cast<int>((static_cast<unsigned long long>(r) * m) >> s);
}
inline void tile_row_magic(int d, unsigned* m, int* s) {
    int l = 0;
    while ((1ll << l) < d) ++l;
    *s = 31 + l;
    *m = static_cast<unsigned>(((1ull << (31 + l)) + static_cast<unsigned long long>(d) - 1) /
                               static_cast<unsigned long long>(d));
}

template <typename T> __device__ __forceinline__ const Phys<T>& phys(const Inst* I);
template <> __device__ __forceinline__ const Phys<float>& phys<float>(const Inst* I) { return I->pf; }
template <> __device__ __forceinline__ const Phys<double>& phys<double>(const Inst* I) { return I->pd; }

// Reciprocal, division and square root of the kernels.  FP32 uses the
// hardware approximations (a couple of ulp, far inside the FP32 error budget
// of the stored populations).  FP64 refines the hardware estimates
// (rcp.approx / rsqrt.approx, accurate to about 2^-22) until only the rounding
// of the last step is left: 1/d by one third-order step (e = 1 - d r,
// r <- r + r (e + e^2), which leaves e^3), sqrt(x) by two steps of
// Goldschmidt's coupled iteration (g -> sqrt(x), h -> 1/(2 sqrt(x)):
// r = 1/2 - g h, g <- g + g r, h <- h + h r).  Both stay within 1 ulp of the
// IEEE-rounded 1/d and sqrt(x) (lbm_fp64_math_check measures this on the
// device); they take fewer FP64 operations than the IEEE sequences, and what
// FP64 does is bound by its pipe.  sqrt keeps sqrt(+-0) = +-0 and NaN for x < 0;
// the FP64 kernels themselves need roots of quotients only (psi_fold_fp64), and
// their divisions are quotient's (lbm_reduce.cuh).
template <typename T> struct Fast;
template <> struct Fast<float> {
    static __device__ __forceinline__ float div(float a, float b) { return __fdividef(a, b); }
    static __device__ __forceinline__ float rcp(float a) { return __fdividef(1.0f, a); }
    static __device__ __forceinline__ float sqrt(float a) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
};
template <> struct Fast<double> {
    // Of 1 / d, where that is infinite or zero; rarely reached, and volatile
    // so that it is not computed ahead of the branch to it.
    static __device__ __forceinline__ double estimate(double d) {
        double r;
        asm volatile("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
        return r;
    }
    static __device__ __forceinline__ double rcp(double d) {
        double r;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
        const double e = fma(-d, r, 1.0);
        return fma(r, fma(e, e, e), r);
    }
    static __device__ __forceinline__ double sqrt(double x) {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        double g = x * y, h = 0.5 * y;
        double r = fma(-g, h, 0.5);
        g = fma(g, r, g);
        h = fma(h, r, h);
        r = fma(-g, h, 0.5);
        g = fma(g, r, g);
        return (__double_as_longlong(x) << 1) == 0 ? x : g;   // +-0: rsqrt is infinite there
    }
};

// psi = sqrt(W / D) = |W| / sqrt(W D): the positive root also beyond the law's
// pole, where W and D are both negative.  1 / sqrt(x) comes from the
// hardware estimate y refined by one third-order step (Householder's
// iteration): with d = 1 - x y^2, y + y d (1/2 + 3/8 d) leaves an error of
// 5/16 d^3, far below the last place from an estimate good to 2^-20; three
// FP64 instructions fewer than two second-order steps (the absolute value is
// an operand's modifier; written in one piece with its product, it leaves the
// schedule as it is without: slabs of 128 x 4 8.92 us a step, 8.97 with fabs()).
// A negative radicand gives NaN (as the square root does), psi(W = 0) = 0.
__device__ __forceinline__ double psi_fold_fp64(double W, double D) {
    const double x = W * D;
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double d = fma(-(x * y), y, 1.0);
    const double r = fma(y * d, fma(d, 0.375, 0.5), y);
    double psi;
    asm("{\n\t.reg .f64 a;\n\tabs.f64 a, %1;\n\tmul.rn.f64 %0, a, %2;\n\t}" : "=d"(psi) : "d"(W), "d"(r));
    return W == 0.0 ? 0.0 : psi;
}

// ---- PTX helpers --------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of the given parity to complete, giving up after
// timeout_ns of wall time.  Returns true when the phase completed.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t timeout_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0 && globaltimer_ns() - t0 > timeout_ns) return false;
    }
}

// Global-memory flags shared between the CTAs of one persistent launch.
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(int* p, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Orders this thread's earlier generic-proxy accesses (the acquire above)
// before its later async-proxy ones (a TMA load of data other CTAs stored).
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

// 3-D tiled TMA load of a box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

}  // namespace lbm

// ---- host-side interfaces between the translation units -----------------
namespace lbm {

struct TileCfg { int bx, by, threads, stages; };

// Fused step (lbm_step.cu).
int step_config_count(int prec);
TileCfg step_config(int prec, int k);
size_t step_smem_bytes(int prec, int k);
cudaError_t step_prepare(int prec, int k);   // sets the dynamic smem attribute
// args: a StepArgs<T> for a context of one lattice (one = true; tile
// coordinates from blockIdx), else a BatchArgs<T> of up to kBatchLaunchMax
// instances, T the context's precision.  ntiles: tiles this launch steps.
cudaError_t step_launch(int prec, int k, const Inst* d_insts, const void* args, bool one, int ntiles, int parity,
                        unsigned long long timeout_ns, cudaStream_t st);
// Multi-step persistent launch of tile configuration k (one box per CTA
// only; false otherwise): args a RunArgs<T>, one = a single instance.  The
// caller has zeroed the step counters, the work counter and the abort flag.
bool run_supported(int prec, int k);
cudaError_t run_launch(int prec, int k, const Inst* d_insts, const void* args, bool one, int ntiles, int nsteps,
                       unsigned long long timeout_ns, cudaStream_t st);

// One lattice held in the shared memory of a thread-block cluster for n
// steps (lbm_cluster.cu; schedule 4): the configuration that this device can
// run for an nx x ny lattice of precision prec (-1: none; sets its kernel's
// attributes), and the launch of that configuration (host: the descriptor),
// which writes the ghost cells of the last time level too.
int cluster_pick(int prec, int nx, int ny);
cudaError_t cluster_run(const Inst& host, int which, int parity, int nsteps, cudaStream_t st);

// Pinned host memory, mapped for every device (lbm_pinned.cu): up to
// kPinnedSmall and up to kPinnedBlock bytes come from slabs of the current
// CUDA context, more straight from the driver.  p NULL when there is none.
// Given back once nothing uses it any more.
constexpr size_t kPinnedSmall = 256, kPinnedBlock = (size_t(1) << 16) + 256;
Pinned pinned_get(size_t bytes);
void pinned_put(const Pinned& b);
// What the driver knows about the memory at p: whether it is pinned host
// memory (and not managed), its address for kernels and the mapped range that
// address is in; known: whether it knows p at all.
struct HostMemory {
    bool known, pinned;
    void* device;
    Span range;
};
HostMemory host_memory(const void* p);

// What a call reads back besides its arrays, written by the device into
// pinned host memory mapped for it: the sums of a reduction with its status
// word, each of which the host watches; or the instance's status word and the
// number of the call whose results these are, written last.
constexpr int kReduceSlots = 8;
struct Reduced {
    double v[kReduceSlots];
    unsigned long long word;   // a reduction's status word
    int status;
    unsigned call;
};
// What a reduction's words hold before their results arrive: a NaN with a
// payload that no arithmetic gives.
constexpr unsigned long long kNoResult = 0x7ff4d1c5a3b29687ull;
// How a kernel gives its results: its last block (by `ticket`, a device word
// that is zero between launches) writes to->call = call once every block's
// writes are visible to the host.  ticket NULL: the status word only (the host
// waits for the stream).
struct Notice {
    Reduced* to;
    unsigned* ticket;
    unsigned call;
};

// Auxiliary kernels (lbm_aux.cu); `host` is the host copy of the descriptor.
// Fields of nx*ny doubles, or floats with f32 (each widened to FP64 exactly).
cudaError_t aux_init(const Inst& host, const Inst* d_inst, const void* rho, const void* ux, const void* uy, bool f32,
                     int parity, cudaStream_t st);
// *word (device) goes to the Notice's status field
cudaError_t aux_fill_ghosts(const Inst& host, const Inst* d_inst, int parity, const Notice& to, const int* word,
                            cudaStream_t st);
// bad |= 1: a density not finite, positive and below rho_max; |= 2: a velocity not finite
cudaError_t aux_check_init(const void* rho, const void* ux, const void* uy, bool f32, long long N, double rho_max,
                           int* bad, cudaStream_t st);
cudaError_t aux_gather_plane(const Inst& host, const Inst* d_inst, int parity, int a, double* out,
                             cudaStream_t st);
// field: 0 rho, 3 psi; rows [y0, y1), written at their place in out
// (row-major, nx per row)
// f32out: floats, each the FP64 value rounded to nearest; `to`: where the
// instance's status word goes and how the host is told
cudaError_t aux_field(const Inst& host, const Inst* d_inst, int parity, int field, int y0, int y1, void* out,
                      bool f32out, const Notice& to, cudaStream_t st);
// rho, ux, uy, psi into out[0..3] (any may be NULL) in one pass; rows and types as above
cudaError_t aux_flow(const Inst& host, const Inst* d_inst, int parity, int y0, int y1, void* const out[4], bool f32out,
                     const Notice& to, cudaStream_t st);
// out: 4 device words (see lbm_fp64_math_check); default stream.
cudaError_t aux_math_check(long long n, double lo, double hi, unsigned long long* out);
// FP64 FMA throughput of the current device (see lbm_fp64_fma_rate).
cudaError_t aux_fp64_fma_rate(int iters, cudaStream_t st, double* flops_per_s, double* seconds);
constexpr int kReduceBlocks = 304;   // rows of partial sums that every context has; larger lattices use their field scratch
// partials: device doubles for the partial sums of `rows` blocks (kReduceSlots each)
cudaError_t aux_measure(const Inst& host, const Inst* d_inst, int parity, double cx, double cy, double r_in,
                        double r_out, bool exact, double* partials, int rows, const Notice& to, cudaStream_t st);
bool aux_measure_again(const double (&sums)[kReduceSlots]);   // with exact set
cudaError_t aux_stats(const Inst& host, const Inst* d_inst, int parity, double* partials, int rows, const Notice& to,
                      cudaStream_t st);

}  // namespace lbm
