// lbm_cluster.cu -- the fused step of a small lattice held in the shared
// memory of one thread-block cluster for all the steps of an lbm_step call
// (schedule 4).
//
// The lattice is cut into strips of BY rows, one per CTA of a cluster of up
// to 16 CTAs (one CTA per SM).  Each CTA keeps two boxes of its strip (all
// nine planes, the strip plus two halo rows above and below and the halo
// columns of the one-step kernel's TMA box) in shared memory: the step's
// input and output time levels.  Per step a CTA
//   1. computes rho and psi (Eq. 10) of its strip and 1-node ring from the
//      input box (the same psi_ring as the one-step kernels);
//   2. collides and streams every owned node into the output box (the same
//      collide_rows, with the output addressed into shared memory);
//   3. writes the periodic images of the output's edge columns (x) into its
//      halo columns, then stores its first two output rows (images included)
//      into the bottom halo rows of the CTA above it and its last two into
//      the top halo rows of the CTA below it (periodic in y through the
//      cluster ranks), in their shared memory (distributed shared memory of
//      the cluster), 16 bytes per store;
//   4. waits at a cluster barrier, after which every output box is complete.
// The per-node arithmetic is that of the one-step kernels on the same box
// contents, so every schedule gives the same bits.  Nothing goes to global
// memory between steps: the populations are read once at the start and
// written once at the end, ghost cells included.  No wait in this kernel spins
// in software: the cluster barrier is the hardware's, every CTA of the cluster
// runs the same number of steps and none leaves early, and a CTA's shared
// memory is only written by the others between two barriers that it takes part
// in.
#include "lbm_host_rules.h"
#include "lbm_step_kernels.cuh"

namespace lbm {
namespace {

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Every thread of every CTA of the cluster: this CTA's shared-memory writes
// (local and remote) before the barrier are visible to all after it.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::
            : "memory");
}
// The address in the shared memory of cluster CTA `rank` of the same
// offset as the local shared-memory address `addr`.
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes: four floats or two doubles.
template <typename T> struct Vec;
template <> struct Vec<float> {
    using type = float4;
    static constexpr int N = 4;
};
template <> struct Vec<double> {
    using type = double2;
    static constexpr int N = 2;
};
template <typename V> __device__ __forceinline__ void st_cluster16(uint32_t addr, const V& v) {
    const uint4 w = reinterpret_cast<const uint4&>(v);
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w)
                 : "memory");
}

template <typename T> struct ClusterArgs {
    Phys<T> P;
    const T* src;      // time level read by the first step
    T* dst;            // time level written by the last step
    long long plane;   // elements per plane of the global arrays
    int pitch;         // elements per row of the global arrays
    int nx, ny, nsteps;
    int* status;
};

template <typename T, int BX, int BY, int NT>
__global__ void __launch_bounds__(NT, 1) k_cluster(const __grid_constant__ ClusterArgs<T> a) {
    using Gm = Geom<T, BX, BY, NT, 1>;
    constexpr int WB = Gm::WB, PB = Gm::PB, HX = Gm::HX;
    constexpr int GXg = Prec<T>::GX;   // ghost columns of the global arrays
    extern __shared__ __align__(1024) unsigned char smem[];
    T* const box0 = reinterpret_cast<T*>(smem);
    T* const box1 = reinterpret_cast<T*>(smem + Gm::buf_stride);
    T* const sp = reinterpret_cast<T*>(smem + 2 * Gm::buf_stride);
    const int tid = threadIdx.x, tx = tid % BX, ty = tid / BX;
    const unsigned rank = cluster_rank(), C = cluster_size();
    const int nx = a.nx, ny = a.ny;
    const int y0 = static_cast<int>(rank) * BY;
    const int h = min(BY, ny - y0);                       // rows of this strip (the host makes it >= 2)
    const int h_last = ny - static_cast<int>(C - 1) * BY;
    const unsigned up = (rank + C - 1) % C, down = (rank + 1) % C;
    const int h_up = up == C - 1 ? h_last : BY;           // rows of the strip above
    const Phys<T>& P = a.P;
    const int interact = P.interact;
    const int path = !interact ? kGeneral : (P.var_visc ? kVisc : (nx == BX && h == BY ? kFast : kRagged));
    const EosRegs<T> E(P);
    const T rho_ref = P.rho_ref;
    // rows move as 16-byte vectors from column -V on, one row of one plane per
    // warp: columns -2 .. nx + 1 carry data
    using Vt = typename Vec<T>::type;
    constexpr int V = Vec<T>::N, kWarps = NT / 32;
    static_assert(HX == V, "a box row starts one vector before its node 0");
    const int nv = (nx + 2 + V - 1) / V + 1, lane = tid & 31, warp = tid >> 5;

    // the input box of the first step: rows y0 - 2 .. y0 + h + 1 and columns
    // -2 .. nx + 1 of the global array (its ghost cells are current)
    for (int k = warp; k < 9 * (h + 4); k += kWarps) {
        const int r = k / 9, q = k - 9 * r;
        const T* const g = a.src + q * a.plane + static_cast<long long>(y0 + r) * a.pitch + (GXg - V);
        T* const o = box0 + q * PB + r * WB;
        for (int v = lane; v < nv; v += 32)   // all of them in flight at once
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(o + v * V)), "l"(g + v * V)
                         : "memory");
    }
    // the other box's padding columns travel with its rows: zeros, as in the global arrays
    for (int e = tid; e < 9 * PB / V; e += NT) reinterpret_cast<uint4*>(box1)[e] = make_uint4(0, 0, 0, 0);
    asm volatile("cp.async.wait_all;" ::: "memory");
    cluster_barrier();   // also: every CTA of the cluster has started before any remote store

    bool bad = false;
#pragma unroll 1
    for (int s = 0; s < a.nsteps; ++s) {
        const T* bi = (s & 1) ? box1 : box0;
        T* bo = (s & 1) ? box0 : box1;
        if (interact) ring_dispatch<Gm, true>(true, P, bi, sp, E, rho_ref, tid, tx, ty);
        __syncthreads();
        // the output of node (x, y) of the strip goes to box row GY + y,
        // column HX + x: collide_rows addresses (y + GY) * pitch + x + GX
        const Regs<T> R(P);
        T* const o = bo - (Gm::GX - HX);
        if (path == kFast)
            bad |= collide_rows<Gm, kFast, false>(bi, sp, P, R, o, PB, WB, 0, 0, nx, h, false, true, tx, ty);
        else if (path == kRagged)
            bad |= collide_rows<Gm, kRagged, false>(bi, sp, P, R, o, PB, WB, 0, 0, nx, h, false, true, tx, ty);
        else if (path == kVisc)
            bad |= collide_rows<Gm, kVisc, false>(bi, sp, P, R, o, PB, WB, 0, 0, nx, h, false, true, tx, ty);
        else
            bad |= collide_rows<Gm, kGeneral, false>(bi, sp, P, R, o, PB, WB, 0, 0, nx, h, false, false, tx, ty);
        __syncthreads();
        // periodic images in x (columns -2, -1 <- nx - 2, nx - 1; nx, nx + 1
        // <- 0, 1), one (row, plane, column) per thread
        for (int k = tid; k < 36 * h; k += NT) {
            const int r = k / 36, e = k - 36 * r, j = e & 3;
            T* const row = bo + (e >> 2) * PB + (GY + r) * WB + HX;
            row[j < 2 ? j - 2 : nx + j - 2] = row[j < 2 ? nx + j - 2 : j - 2];
        }
        __syncthreads();
        // the edge rows with their images to the neighbours' halo rows, one
        // (row k < 4, plane) per warp: rows GY, GY + 1 to rows GY + h_up, GY +
        // h_up + 1 of the CTA above, rows GY + h - 2, GY + h - 1 to rows 0, 1 of
        // the CTA below.  (A lane that forms an image itself makes its whole
        // warp wait for the gather: 1290 clocks per step instead of 350.)
        auto edge_row = [&](int k, const T*& from, uint32_t& to) {
            const int row = k / 9, q = k - 9 * row;
            from = bo + q * PB + (row < 2 ? GY + row : GY + h - 4 + row) * WB;
            to = cluster_map(smem_u32(bo + q * PB + (row < 2 ? GY + h_up + row : row - 2) * WB), row < 2 ? up : down);
        };
        if (lane < nv) {
            constexpr int kPairs = (36 + kWarps - 1) / kWarps;   // loaded together, then sent
            Vt w[kPairs];
            uint32_t to[kPairs];
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                const T* from;
                if (warp + i * kWarps < 36) {
                    edge_row(warp + i * kWarps, from, to[i]);
                    w[i] = *reinterpret_cast<const Vt*>(from + lane * V);
                }
            }
#pragma unroll
            for (int i = 0; i < kPairs; ++i)
                if (warp + i * kWarps < 36) st_cluster16(to[i] + lane * 16u, w[i]);
        }
        const int rest = nv - 32;   // vectors beyond the lanes: few, one per thread
        for (int k = tid; k < 36 * rest; k += NT) {
            const T* from;
            uint32_t to;
            const int v = 32 + k / 36;
            edge_row(k % 36, from, to);
            st_cluster16(to + v * 16u, *reinterpret_cast<const Vt*>(from + v * V));
        }
        cluster_barrier();
    }

    // the last output box's strip to the global array, with its ghost cells:
    // the strip's rows carry their x images, and the lattice's first and last
    // two rows also go to the ghost rows opposite
    const T* fin = (a.nsteps & 1) ? box1 : box0;
    const long long wrap = static_cast<long long>(ny) * a.pitch;
    for (int k = warp; k < 9 * h; k += kWarps) {
        const int r = k / 9, q = k - 9 * r, y = y0 + r;
        const T* const g = fin + q * PB + (GY + r) * WB;
        T* const d = a.dst + q * a.plane + static_cast<long long>(y + GY) * a.pitch + (GXg - V);
        for (int v = lane; v < nv; v += 32) {
            const Vt w = *reinterpret_cast<const Vt*>(g + v * V);
            *reinterpret_cast<Vt*>(d + v * V) = w;
            if (y < 2) *reinterpret_cast<Vt*>(d + wrap + v * V) = w;
            if (y >= ny - 2) *reinterpret_cast<Vt*>(d - wrap + v * V) = w;
        }
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(a.status, ST_UNSTABLE);
}

template <typename T> ClusterArgs<T> cluster_args(const Inst& h, int parity, int nsteps) {
    ClusterArgs<T> a;
    if constexpr (sizeof(T) == 4) a.P = h.pf;
    else a.P = h.pd;
    a.src = static_cast<const T*>(h.pop[parity]);
    a.dst = static_cast<T*>(h.pop[parity ^ (nsteps & 1)]);
    a.plane = h.plane;
    a.pitch = h.pitch;
    a.nx = h.nx;
    a.ny = h.ny;
    a.nsteps = nsteps;
    a.status = h.status;
    return a;
}

// A cluster configuration: strips of BY rows of at most BX nodes, NT threads.
template <typename T, int BX, int BY, int NT> struct ClusterCfg {
    using Gm = Geom<T, BX, BY, NT, 1>;
    static constexpr size_t smem = 2 * Gm::buf_stride + Gm::psi_stride;
    static_assert(smem <= 232448, "two boxes and the psi tile must fit in a CTA's shared memory");
    static constexpr ClusterShape shape = {BX, BY};
    // the launch of one cluster of C CTAs
    static void config(int C, cudaStream_t st, cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr) {
        cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(C));
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = static_cast<unsigned>(C);
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    // whether the device can hold a cluster of this lattice's CTAs at all; sets
    // the kernel's attributes, which every later launch on the device needs
    static bool launchable(int ny) {
        const auto fn = &k_cluster<T, BX, BY, NT>;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return false;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        int n = 0;
        config(shape.ctas(ny), nullptr, cfg, attr);
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, &k_cluster<T, BX, BY, NT>, &cfg);
        if (e != cudaSuccess) cudaGetLastError();   // not the next launch's error
        return e == cudaSuccess && n > 0;
    }
    static cudaError_t run(const Inst& h, int parity, int nsteps, cudaStream_t st) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        config(shape.ctas(h.ny), st, cfg, attr);
        return cudaLaunchKernelEx(&cfg, &k_cluster<T, BX, BY, NT>, cluster_args<T>(h, parity, nsteps));
    }
};

// One node per thread.  FP32, up to 64 nodes wide: strips of 4 rows up to 64
// high, of 8 up to 128, else of 16, so that a small lattice is spread over as
// many SMs as a cluster may have (64^2: 16 CTAs of 256 threads 1.41 us per
// step, four CTAs of 1024 threads 2.85 us; 64 x 100: 1.63 and 2.85); up to
// 128 wide: strips of 8 rows.  FP64, bound by its FP64 pipe, likewise: 4 rows
// up to 64 high, else 8, up to 64 nodes wide.  Clocks of a 64^2 FP32 step:
// psi ring 610, collision 590, images and edge rows 590, cluster barrier with
// the remote stores' arrival 1000.
template <class... Cfg> struct ClusterTable {
    static constexpr int count = sizeof...(Cfg);
    static constexpr ClusterShape shapes[] = {Cfg::shape...};
    static int pick(int nx, int ny) {
        static constexpr bool (*launchable[])(int) = {&Cfg::launchable...};
        return pick_cluster(shapes, count, nx, ny, [&](int k) { return launchable[k](ny); });
    }
    static cudaError_t run(int which, const Inst& h, int parity, int nsteps, cudaStream_t st) {
        static constexpr cudaError_t (*runs[])(const Inst&, int, int, cudaStream_t) = {&Cfg::run...};
        return which >= 0 && which < count ? runs[which](h, parity, nsteps, st) : cudaErrorInvalidValue;
    }
};
using ClusterF32 = ClusterTable<ClusterCfg<float, 64, 4, 256>, ClusterCfg<float, 64, 8, 512>,
                                ClusterCfg<float, 64, 16, 1024>, ClusterCfg<float, 128, 8, 1024>>;
using ClusterF64 = ClusterTable<ClusterCfg<double, 64, 4, 256>, ClusterCfg<double, 64, 8, 512>>;

}  // namespace

int cluster_pick(int prec, int nx, int ny) {
    return prec == LBM_FP32 ? ClusterF32::pick(nx, ny) : ClusterF64::pick(nx, ny);
}

cudaError_t cluster_run(const Inst& h, int which, int parity, int nsteps, cudaStream_t st) {
    if (nsteps <= 0) return cudaSuccess;
    return h.prec == LBM_FP32 ? ClusterF32::run(which, h, parity, nsteps, st)
                              : ClusterF64::run(which, h, parity, nsteps, st);
}

}  // namespace lbm
