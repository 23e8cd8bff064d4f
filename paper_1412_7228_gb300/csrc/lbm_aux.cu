// lbm_aux.cu -- kernels around the fused step: initial equilibrium, ghost
// images, read-back of populations and macroscopic fields, and the FP64
// reductions behind Laplace's law (Eq. 22) and the run statistics.
// None of these is on the per-step path.
#include <type_traits>

#include "lbm_internal.cuh"
#include "lbm_init.h"
#include "lbm_reduce.cuh"

namespace lbm {
namespace {

constexpr int kThreads = 256;

// Lattice weights t_a of the D2Q9 equilibrium (4/9, 1/9, 1/36).
__device__ __forceinline__ double tw(int a) { return a == 0 ? 4.0 / 9.0 : (a < 5 ? 1.0 / 9.0 : 1.0 / 36.0); }

template <typename T> __device__ __forceinline__ T* popk(const Inst* I, int parity) {
    return static_cast<T*>(I->pop[parity]);
}

// Element (a, x, y) of a time level; x in [-GX, pitch-GX), y in [-2, ny+2).
template <typename T> __device__ __forceinline__ long long at(const Inst* I, int a, int x, int y) {
    return a * I->plane + static_cast<long long>(y + GY) * I->pitch + (x + Prec<T>::GX);
}

// Node loops over a lattice: rows y by blockIdx.y, columns x by the
// threads of blockIdx.x (grid from grid_2d), so that no thread divides by
// the lattice width.
#define LBM_FOR_NODES(nx, ny)                                      \
    for (int y = blockIdx.y; y < (ny); y += gridDim.y)             \
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < (nx); x += gridDim.x * blockDim.x)

// ---- initial state: f_a(z) = f_eq,a(rho(z), u(z)); pull storage keeps it at z - e_a
// REST: no velocity field given (u = 0), where the equilibrium's velocity
// terms are exact zeros and the deviation is t_a (rho - rho_ref): FP64
// keeps the FP64 products; FP32 rounds rho - rho_ref (formed in FP64, so
// that no digit of a small difference is lost) to FP32 once and multiplies
// by the weights in FP32 (within 1.5 ulp of the correctly rounded value, and
// two FP64 operations per node instead of seven: GB300's FP64 pipe would
// otherwise bound the initialisation).  With a velocity the nine
// values share the products of r, u and v: 33 FP64 instructions instead of
// about 80 (FP32 lattice, 1531 x 1117 in bands: 38.8 -> 22.7 us a band).
template <typename T, bool REST, typename R>
__device__ __forceinline__ void equilibrium(double rr, R rho, R ux, R uy, T (&f)[9]) {
    const double d = static_cast<double>(rho) - rr;
    constexpr double t0 = 4.0 / 9.0, t1 = 1.0 / 9.0, t5 = 1.0 / 36.0;
    if constexpr (REST) {
        T t[3];
        if constexpr (sizeof(T) == 4) {
            const float df = static_cast<float>(d);
            t[0] = __fmul_rn(4.0f / 9.0f, df);
            t[1] = __fmul_rn(1.0f / 9.0f, df);
            t[2] = __fmul_rn(1.0f / 36.0f, df);
        } else {
            t[0] = t0 * d;
            t[1] = t1 * d;
            t[2] = t5 * d;
        }
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = t[a == 0 ? 0 : (a < 5 ? 1 : 2)];
    } else {
        // t_a [(r - rr) + r (3 e.v + 4.5 (e.v)^2 - 1.5 v^2)], v = (u, v)
        const double r = rho, u = ux, v = uy, ru = r * u, rv = r * v, uu = ru * u, vv = rv * v, uv = ru * v;
        const double s = uu + vv, B = fma(-1.5, s, d), X = fma(4.5, uu, B), Y = fma(4.5, vv, B);
        const double D = fma(4.5, s, B), P = fma(9.0, uv, D), M = fma(-9.0, uv, D), sp = ru + rv, sm = ru - rv;
        f[0] = static_cast<T>(t0 * B);
        f[1] = static_cast<T>(t1 * fma(3.0, ru, X));
        f[3] = static_cast<T>(t1 * fma(-3.0, ru, X));
        f[2] = static_cast<T>(t1 * fma(3.0, rv, Y));
        f[4] = static_cast<T>(t1 * fma(-3.0, rv, Y));
        f[5] = static_cast<T>(t5 * fma(3.0, sp, P));
        f[7] = static_cast<T>(t5 * fma(-3.0, sp, P));
        f[8] = static_cast<T>(t5 * fma(3.0, sm, M));
        f[6] = static_cast<T>(t5 * fma(-3.0, sm, M));
    }
}

// The checks of an initial field, on the device: bit 1 of *bad when a
// density is not finite, not positive or not below rho_max, bit 2 when a
// velocity is not finite (the caller has zeroed *bad).  On the bit patterns,
// as integers (no FP64 work): for rho_max > 0, 0 < r < rho_max with r finite
// is 0 < bits(r) < bits(top), top = rho_max in FP64, or for FP32 fields the
// smallest float not below rho_max (positive values order as their patterns;
// negatives and -0 have the sign bit, NaN and inf patterns lie above every
// finite value); finite is an exponent field below all ones.
__device__ __forceinline__ long long bits_of(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ long long bits_of(float v) { return __float_as_int(v); }
template <typename R> __host__ __device__ constexpr long long exp_mask() {
    return sizeof(R) == 8 ? 0x7ff0000000000000ll : 0x7f800000ll;
}
__device__ __forceinline__ long long top_bits(double rho_max, double) { return bits_of(rho_max); }
__device__ __forceinline__ long long top_bits(double rho_max, float) { return bits_of(__double2float_ru(rho_max)); }
template <typename R> struct FieldCheck {
    long long top;
    int b = 0;
    __device__ __forceinline__ explicit FieldCheck(double rho_max) : top(top_bits(rho_max, R(0))) {}
    __device__ __forceinline__ void density(R v) {
        const long long r = bits_of(v);
        if (!(r > 0 && r < top)) b |= 1;
    }
    __device__ __forceinline__ void velocity(R v) {
        constexpr long long kExp = exp_mask<R>();
        if ((bits_of(v) & kExp) == kExp) b |= 2;
    }
    __device__ __forceinline__ void report(int* bad) {   // every lane of the warp
        b = __reduce_or_sync(0xffffffffu, b);
        if (b && (threadIdx.x & 31) == 0) atomicOr(bad, b);
    }
};

// Rows [y0, y1) of the field; rho, ux and uy index the whole field, in device
// memory or in pinned host memory (each value is read once, so the field
// need not be copied first).  bad != NULL: the values are checked on the way.
template <typename T, bool REST, typename R>
__global__ void k_init(const Inst* __restrict__ I, const R* __restrict__ rho, const R* __restrict__ ux,
                       const R* __restrict__ uy, int parity, int y0, int y1, double rho_max, int* bad) {
    const int nx = I->nx, ny = I->ny;
    T* p = popk<T>(I, parity);
    const double rr = static_cast<double>(phys<T>(I).rho_ref);
    FieldCheck<R> check(rho_max);
    for (int y = y0 + static_cast<int>(blockIdx.y); y < y1; y += gridDim.y)
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nx; x += gridDim.x * blockDim.x) {
            const long long i = static_cast<long long>(y) * nx + x;
            const R r = rho[i], u = !REST && ux ? ux[i] : R(0), v = !REST && uy ? uy[i] : R(0);
            check.density(r);
            if (!REST) {
                check.velocity(u);
                check.velocity(v);
            }
            T f[9];
            equilibrium<T, REST>(rr, r, u, v, f);
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                int xs = x - cx(a), ys = y - cy(a);
                xs = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
                ys = ys < 0 ? ys + ny : (ys >= ny ? ys - ny : ys);
                p[at<T>(I, a, xs, ys)] = f[a];
            }
        }
    __syncwarp();
    if (bad) check.report(bad);
}

template <typename R>
__global__ void k_check_init(const R* __restrict__ rho, const R* __restrict__ ux, const R* __restrict__ uy,
                             long long N, double rho_max, int* bad) {
    FieldCheck<R> check(rho_max);
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < N;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        check.density(rho[i]);
        if (ux) check.velocity(ux[i]);
        if (uy) check.velocity(uy[i]);
    }
    __syncwarp();
    check.report(bad);
}

// The block's writes are done: the last block tells the host (Notice).
__device__ __forceinline__ void notify(const Notice& to) {
    if (!to.ticket) return;
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (atomicAdd(to.ticket, 1u) != gridDim.x * gridDim.y - 1) return;
    *to.ticket = 0;
    __threadfence_system();
    *static_cast<volatile unsigned*>(&to.to->call) = to.call;
}
// Ghost cells x in [-2,0) U [nx,nx+2), y in [-2,0) U [ny,ny+2) of every
// plane, and only those: per plane the rows y = -2, -1, ny, ny + 1 over
// x in [-2, nx + 2) (4 (nx + 4) cells), then the columns x = -2, -1, nx,
// nx + 1 over y in [0, ny) (4 ny cells).  Each copies its periodic image
// inside the lattice.  With a Notice, *word goes to its status field.
template <typename T>
__global__ void k_ghosts(const Inst* __restrict__ I, int parity, Notice to, const int* __restrict__ word) {
    if (to.ticket && blockIdx.x == 0 && threadIdx.x == 0) to.to->status = *word;
    const int nx = I->nx, ny = I->ny;
    const int W = nx + 4, per = 4 * W + 4 * ny;
    const long long M = 9ll * per;
    T* p = popk<T>(I, parity);
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < M;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int a = static_cast<int>(i / per);
        const int r = static_cast<int>(i - static_cast<long long>(a) * per);
        int x, y;
        if (r < 4 * W) {
            const int row = r / W;
            x = r - row * W - 2;
            y = row < 2 ? row - 2 : ny + row - 2;
        } else {
            const int q = r - 4 * W, col = q / ny;
            y = q - col * ny;
            x = col < 2 ? col - 2 : nx + col - 2;
        }
        const int xs = ((x % nx) + nx) % nx, ys = ((y % ny) + ny) % ny;
        p[at<T>(I, a, x, y)] = p[at<T>(I, a, xs, ys)];
    }
    notify(to);
}

// f_a(z, t) = pop_a(z - e_a) + t_a rho_ref, for one plane a.
template <typename T>
__global__ void k_gather(const Inst* __restrict__ I, int parity, int a, double* __restrict__ out) {
    const int nx = I->nx, ny = I->ny;
    const T* p = popk<T>(I, parity);
    const double off = tw(a) * static_cast<double>(phys<T>(I).rho_ref);
    const int ex = cx(a), ey = cy(a);
    LBM_FOR_NODES(nx, ny) {
        out[static_cast<long long>(y) * nx + x] = static_cast<double>(p[at<T>(I, a, x - ex, y - ey)]) + off;
    }
}

// The nine populations pulled by node (x, y), x in [-1, nx], y in [-1, ny].
template <typename T> __device__ __forceinline__ void node_pops(const Inst* I, const T* p, int x, int y, T (&v)[9]) {
#pragma unroll
    for (int a = 0; a < 9; ++a) v[a] = p[at<T>(I, a, x - cx(a), y - cy(a))];
}

// A float as a double, by moving its bits: the conversion instruction holds
// the FP64 pipe as long as an addition.  A denormal is first made normal (by an
// exact product with 2^64); the value is below infinity.
__device__ __forceinline__ double widen(float v) {
    const bool tiny = (__float_as_uint(v) & 0x7f800000u) == 0;
    const unsigned u = __float_as_uint(tiny ? __fmul_rn(v, 0x1p64f) : v), mag = u & 0x7fffffffu;
    const unsigned hi = mag ? (mag >> 3) + (tiny ? 0x38000000u - (64u << 20) : 0x38000000u) : 0u;
    return __hiloint2double(static_cast<int>((u & 0x80000000u) | hi), static_cast<int>(u << 29));
}

// Sum of N floats in FP64 accuracy with three FP64 additions: the sum as an
// unevaluated triple hi + lo + lo2 (Knuth's TwoSum gives the exact error of
// each addition; the errors' own sum is kept the same way), within 2^-69 of
// the largest partial sum, closer than adding the N values one after another
// in FP64.  About 13 FP32 operations per value, which GB300 issues at 64
// times the rate of FP64 ones.  A sum that leaves FP32's range (an unstable
// lattice) is formed in FP64.
template <int N> __device__ __forceinline__ double sum_f32(const float (&v)[N], double plus) {
    float hi = v[0], lo = 0.0f, lo2 = 0.0f;
    auto two_sum = [](float a, float b, float& err) {
        const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
        err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
        return s;
    };
#pragma unroll
    for (int k = 1; k < N; ++k) {
        float e, e2;
        hi = two_sum(hi, v[k], e);
        lo = two_sum(lo, e, e2);
        lo2 = __fadd_rn(lo2, e2);
    }
    if (!(fabsf(hi) < 3.0e38f)) {
        double r = 0.0;
        for (int k = 0; k < N; ++k) r += static_cast<double>(v[k]);
        return r + plus;
    }
    return (widen(hi) + plus) + (widen(lo) + widen(lo2));
}

// rho of a node from its nine populations.
__device__ __forceinline__ double node_rho(const Inst* I, const float (&v)[9]) {
    return sum_f32<9>(v, static_cast<double>(I->pf.rho_ref));
}
__device__ __forceinline__ double node_rho(const Inst* I, const double (&v)[9]) {
    double r = 0.0;
#pragma unroll
    for (int a = 0; a < 9; ++a) r += v[a];
    return r + I->pd.rho_ref;
}
template <typename T> __device__ __forceinline__ double node_rho(const Inst* I, const T* p, int x, int y) {
    T v[9];
    node_pops(I, p, x, y, v);
    return node_rho(I, v);
}
// momentum sum f e
__device__ __forceinline__ void node_j(const float (&v)[9], double& jx, double& jy) {
    const float sx[6] = {v[1], -v[3], v[5], -v[6], -v[7], v[8]}, sy[6] = {v[2], -v[4], v[5], v[6], -v[7], -v[8]};
    jx = sum_f32<6>(sx, 0.0);
    jy = sum_f32<6>(sy, 0.0);
}
__device__ __forceinline__ void node_j(const double (&v)[9], double& jx, double& jy) {
    jx = v[1] - v[3] + v[5] - v[6] - v[7] + v[8];
    jy = v[2] - v[4] + v[5] + v[6] - v[7] - v[8];
}

// Tiles of the kernels that need the force (velocity fields, statistics):
// psi of the tile and its 1-node ring (periodic) goes to shared memory once,
// so a node costs 1.25 densities and psi instead of nine, and 64 FP64
// instructions (FP32 velocities; statistics 76) instead of 700 (the FP64 pipe is the bound: 19 clocks of an
// SM per warp instruction).  32 x 16 nodes: two per thread, a ring of 612
// nodes in 20 warp passes for 16 of the tile's own.  FP32 statistics of
// 1024^2: 1113 -> 177 us per call, of 256^2: 149 -> 27; the two velocity
// components of 1531 x 1117: 2 x 1709 -> 277 us, rho and psi with them.
// Lattices that leave SMs idle (up to 128^2) take 32 x 4 tiles of 128 threads,
// whose larger ring costs less than the longer chain (statistics of 64^2: 20.8
// us on the device with 32 x 16 tiles, 11.8 with 32 x 4).
constexpr int kFlowX = 32, kFlowW = kFlowX + 2;
template <int NT> struct FlowTile {
    static constexpr int Y = NT == 128 ? 4 : 16, H = Y + 2;
    double psi[H][kFlowW], h[H][kFlowW], rho[H][kFlowW];   // h: hF psi^2, as in the step kernels
};

// rho, velocity (rho u = sum f e + F/2, F of Eq. 9) and psi of the nodes
// of tile (x0, y0), rows below y1, given to use(x, y, rho, ux, uy, psi) by
// the thread that owns each; every thread of the block (NT) calls it.
template <int NT, typename T, typename Use>
__device__ __forceinline__ void flow_tile(const Inst* I, const T* p, int x0, int y0, int y1, FlowTile<NT>& S, Use use) {
    constexpr int kFlowY = FlowTile<NT>::Y, kFlowH = FlowTile<NT>::H;
    const Phys<double>& P = I->pd;
    const int nx = I->nx, ny = I->ny, interact = P.interact;
    const int tid = threadIdx.x;
    if (interact) {
        const LawFp64 law(P, true);
        const int w = min(kFlowX, nx - x0) + 2, h = min(kFlowY, y1 - y0) + 2;
        for (int e = tid; e < kFlowW * kFlowH; e += NT) {
            const int j = e / kFlowW, i = e - j * kFlowW;
            if (i >= w || j >= h) continue;
            int x = x0 + i - 1, y = y0 + j - 1;
            x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
            y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
            const double r = node_rho<T>(I, p, x, y);
            const double ps = law.psi(r);
            S.rho[j][i] = r;
            S.psi[j][i] = ps;
            S.h[j][i] = (P.hF * ps) * ps;
        }
        __syncthreads();
    }
    const double cF = P.cF;
    const int i = tid % kFlowX + 1, x = x0 + i - 1;
    for (int j = tid / kFlowX + 1; j <= kFlowY; j += NT / kFlowX) {
        const int y = y0 + j - 1;
        if (x >= nx || y >= y1) continue;
        T v[9];
        node_pops(I, p, x, y, v);
        const double r = interact ? S.rho[j][i] : node_rho(I, v);
        double jx, jy, ps = 0.0;
        node_j(v, jx, jy);
        if (interact) {
            // Eq. 9 with the weights 12 w_a (4 on the axes, 1 on the
            // diagonals) over g_a = -(G/12) [(1-A) psi psi_a + (A/2) psi_a^2]
            ps = S.psi[j][i];
            const double c = cF * ps;
            auto g = [&](int dj, int di) { return fma(c, S.psi[j + dj][i + di], S.h[j + dj][i + di]); };
            const double a57 = g(1, 1) - g(-1, -1), a86 = g(-1, 1) - g(1, -1);
            jx = fma(0.5, fma(4.0, g(0, 1) - g(0, -1), a57 + a86), jx);
            jy = fma(0.5, fma(4.0, g(1, 0) - g(-1, 0), a57 - a86), jy);
        }
        const double inv = Fast<double>::rcp(r);
        use(x, y, r, quotient_any(jx, inv, r), quotient_any(jy, inv, r), ps);
    }
    if (interact) __syncthreads();   // before the next tile's psi
}

// rho or psi of the nodes, one field per launch (FIELD 0 rho, 3 psi): the
// density read-back keeps the registers of a plain gather.  Rows [y0, y1) of
// the field, at their place in out (row-major nx x ny).
template <typename T, int FIELD, typename O>
__global__ void k_field(const Inst* __restrict__ I, int parity, int y0, int y1, O* __restrict__ out,
                        Notice to) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) to.to->status = *I->status;
    const int nx = I->nx;
    const T* p = popk<T>(I, parity);
    const LawFp64 law(I->pd, true);
    for (int y = y0 + static_cast<int>(blockIdx.y); y < y1; y += gridDim.y)
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nx; x += gridDim.x * blockDim.x) {
            const double r = node_rho<T>(I, p, x, y);
            double v = r;
            if constexpr (FIELD == 3) v = I->pd.interact ? law.psi(r) : 0.0;
            out[static_cast<long long>(y) * nx + x] = static_cast<O>(v);
        }
    notify(to);
}

// The velocity components and, where asked for, rho and psi of rows [y0, y1)
// in one pass (any output may be NULL).
template <int NT, typename T, typename O>
__global__ void __launch_bounds__(NT) k_flow(const Inst* __restrict__ I, int parity, int y0, int y1,
                                                   O* __restrict__ rho, O* __restrict__ ux, O* __restrict__ uy,
                                                   O* __restrict__ psi, Notice to) {
    __shared__ FlowTile<NT> S;
    constexpr int kFlowY = FlowTile<NT>::Y;
    if (blockIdx.x == 0 && threadIdx.x == 0) to.to->status = *I->status;
    const int nx = I->nx, tiles_x = (nx + kFlowX - 1) / kFlowX, tiles = tiles_x * ((y1 - y0 + kFlowY - 1) / kFlowY);
    const T* p = popk<T>(I, parity);
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int ty = t / tiles_x;
        flow_tile<NT, T>(I, p, (t - ty * tiles_x) * kFlowX, y0 + ty * kFlowY, y1, S,
                     [&](int x, int y, double r, double u, double w, double ps) {
                         const long long i = static_cast<long long>(y) * nx + x;
                         if (rho) rho[i] = static_cast<O>(r);
                         if (ux) ux[i] = static_cast<O>(u);
                         if (uy) uy[i] = static_cast<O>(w);
                         if (psi) psi[i] = static_cast<O>(ps);
                     });
    }
    notify(to);
}

// The results of a reduction and the status word, by threads 0..7 of the
// last block.  Each is one word, which the host has set to kNoResult before
// and watches for itself, so none waits for another to be visible (a fence to
// the host's memory takes a microsecond).
__device__ __forceinline__ void give(const Notice& to, double total, const Inst* I) {
    volatile Reduced* const r = to.to;
    r->v[threadIdx.x] = total;
    if (threadIdx.x == 0) r->word = static_cast<unsigned>(*I->status);
}

// ---- FP64 reductions (lbm_reduce.cuh) -------------------------------------
// Sums for Laplace's law (LaplaceSums); p = p_EOS(rho) (equal to
// rho/3 + G psi^2/2, Eq. 10).  The last block puts the totals and the
// instance's status into mapped host memory: the call needs no second launch,
// no copy and no wait for the stream.  About 22 FP64 instructions per node (nine
// additions in FP64, the square root and the divisions by the lattice's size
// are gone).  Per call, FP32: 256^2 88 -> 18 us, 1024^2 236 -> 72 us.
template <typename T, bool EXACT>
__global__ void __launch_bounds__(kLapThreads) k_measure(const Inst* __restrict__ I, int parity, Discs D, int rpt,
                                                       double* __restrict__ partials, Notice to) {
    __shared__ AxisTable A;
    const T* p = popk<T>(I, parity);
    LaplaceSums<EXACT> L;
    laplace_tiles(L, LawFp64(I->pd, false), D, I->nx, I->ny, rpt, A,
                  [&](int x, int y) { return node_rho<T>(I, p, x, y); });
    double total;
    if (grid_sum8<kLapThreads>(L.v, -1, 0.0, partials, to.ticket, &total)) give(to, total, I);
}

// {mass, sum rho u_x, sum rho u_y, sum rho |u|^2 / 2, max |u|, 0, 0, 0}
template <int NT, typename T>
__global__ void __launch_bounds__(NT) k_stats(const Inst* __restrict__ I, int parity, double* __restrict__ partials,
                                                     Notice to) {
    __shared__ FlowTile<NT> S;
    constexpr int kFlowY = FlowTile<NT>::Y;
    const int nx = I->nx, ny = I->ny;
    const int tiles_x = (nx + kFlowX - 1) / kFlowX, tiles = tiles_x * ((ny + kFlowY - 1) / kFlowY);
    const T* p = popk<T>(I, parity);
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0}, most = 0.0;   // most: max |u|^2 (the root is monotone)
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int ty = t / tiles_x;
        flow_tile<NT, T>(I, p, (t - ty * tiles_x) * kFlowX, ty * kFlowY, ny, S,
                     [&](int, int, double r, double u, double w, double) {
                         const double u2 = u * u + w * w;
                         v[0] += r;
                         v[1] += r * u;
                         v[2] += r * w;
                         v[3] += 0.5 * r * u2;
                         most = fmax(most, u2);
                     });
    }
    double total;
    if (grid_sum8<NT>(v, 4, most, partials, to.ticket, &total)) give(to, threadIdx.x == 4 ? sqrt(total) : total, I);
}

int grid_for(long long n) {
    long long b = (n + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    if (b > 8 * kReduceBlocks) b = 8 * kReduceBlocks;
    return static_cast<int>(b);
}

// Grid of the node loops (LBM_FOR_NODES): up to 8 blocks across a row, the
// rest down the rows, 8 * kReduceBlocks blocks at most.
dim3 grid_2d(int nx, int ny) {
    int gx = (nx + kThreads - 1) / kThreads;
    if (gx > 8) gx = 8;
    if (gx < 1) gx = 1;
    int gy = 8 * kReduceBlocks / gx;
    if (gy > ny) gy = ny;
    if (gy < 1) gy = 1;
    return dim3(static_cast<unsigned>(gx), static_cast<unsigned>(gy));
}

// ---- FP64 reciprocal, division and square root against IEEE --------------
// Distance in units in the last place; values of opposite sign or NaN count
// as infinitely far.
__device__ __forceinline__ unsigned long long ulp_distance(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    if (x == y) return 0;
    if (!(a == a) || !(b == b) || ((x ^ y) < 0)) return ~0ull;
    return static_cast<unsigned long long>(x > y ? x - y : y - x);
}

// out[0..2]: largest distance of Fast<double>::rcp(d), quotient(a, rcp(d), d)
// and Fast<double>::sqrt(d) from 1/d, a/d, sqrt(d) (IEEE-rounded: this file keeps nvcc's default
// -prec-div and -prec-sqrt) over n values of d spread evenly over [lo, hi],
// a in [0.37, 0.87); out[3] = 1 if sqrt keeps +0, -0 and gives NaN for -1.
__global__ void k_math_check(long long n, double lo, double hi, unsigned long long* out) {
    unsigned long long m0 = 0, m1 = 0, m2 = 0;
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n; i += stride) {
        const double d = lo + (hi - lo) * (static_cast<double>(i) / static_cast<double>(n));
        const double a = 0.37 + 0.5 * static_cast<double>((i * 2654435761ll) & 0xffff) / 65536.0;
        const double inv = Fast<double>::rcp(d);
        m0 = max(m0, ulp_distance(inv, 1.0 / d));
        m1 = max(m1, ulp_distance(quotient(a, inv, d), a / d));
        m2 = max(m2, ulp_distance(Fast<double>::sqrt(d), sqrt(d)));
    }
    atomicMax(&out[0], m0);
    atomicMax(&out[1], m1);
    atomicMax(&out[2], m2);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double pz = Fast<double>::sqrt(0.0), nz = Fast<double>::sqrt(-0.0), neg = Fast<double>::sqrt(-1.0);
        out[3] = (__double_as_longlong(pz) == 0 && __double_as_longlong(nz) == __double_as_longlong(-0.0) &&
                  !(neg == neg))
                     ? 1ull
                     : 0ull;
    }
}

// FP64 fused multiply-add throughput: every thread runs kFmaChains
// independent chains x <- x m + c (m < 1, so x stays finite) for `iters`
// iterations.  The chains' sum is compared with a value it cannot take, so
// the compiler keeps every FMA; nothing is stored.
constexpr int kFmaChains = 8;
constexpr int kFmaThreads = 256;
__device__ double g_fma_sink;
__global__ void __launch_bounds__(kFmaThreads) k_fp64_fma(int iters, double m, double c) {
    double x[kFmaChains];
#pragma unroll
    for (int k = 0; k < kFmaChains; ++k) x[k] = 1e-3 * threadIdx.x + k;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < kFmaChains; ++k) x[k] = fma(x[k], m, c);
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kFmaChains; ++k) s += x[k];
    if (s == -1.0) g_fma_sink = s;
}

}  // namespace

cudaError_t aux_fp64_fma_rate(int iters, cudaStream_t st, double* flops_per_s, double* seconds) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int blocks = sms * (2048 / kFmaThreads);   // every SM full
    cudaEvent_t e0, e1;
    if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
    if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
        cudaEventDestroy(e0);
        return e;
    }
    float best = 0.0f;
    for (int r = 0; r < 4 && e == cudaSuccess; ++r) {   // the first launch warms up
        e = cudaEventRecord(e0, st);
        if (e == cudaSuccess) {
            k_fp64_fma<<<blocks, kFmaThreads, 0, st>>>(iters, 0.999, 1e-3);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaEventRecord(e1, st);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && r > 0 && (best == 0.0f || ms < best)) best = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return e;
    const double flops = 2.0 * blocks * kFmaThreads * static_cast<double>(kFmaChains) * iters;
    *seconds = best * 1e-3;
    *flops_per_s = flops / (*seconds);
    return cudaSuccess;
}

template <typename R>
cudaError_t init_rows_t(const Inst& h, const Inst* d, const R* rho, const R* ux, const R* uy, int parity, int y0,
                        int y1, double rho_max, int* bad, cudaStream_t st) {
    const dim3 g = grid_2d(h.nx, y1 - y0);
    const bool rest = !ux && !uy;
    auto go = [&](auto k) { k<<<g, kThreads, 0, st>>>(d, rho, ux, uy, parity, y0, y1, rho_max, bad); };
    if (h.prec == LBM_FP32) rest ? go(k_init<float, true, R>) : go(k_init<float, false, R>);
    else rest ? go(k_init<double, true, R>) : go(k_init<double, false, R>);
    return cudaGetLastError();
}

cudaError_t aux_init(const Inst& h, const Inst* d, const void* rho, const void* ux, const void* uy, bool f32,
                     int parity, cudaStream_t st) {
    const cudaError_t e = aux_init_rows(h, d, rho, ux, uy, f32, parity, 0, h.ny, 0.0, nullptr, st);
    return e != cudaSuccess ? e : aux_fill_ghosts(h, d, parity, Notice{}, nullptr, st);
}

cudaError_t aux_init_rows(const Inst& h, const Inst* d, const void* rho, const void* ux, const void* uy, bool f32,
                          int parity, int y0, int y1, double rho_max, int* bad, cudaStream_t st) {
    if (y0 < 0 || y1 > h.ny || y0 >= y1) return cudaErrorInvalidValue;
    if (f32)
        return init_rows_t(h, d, static_cast<const float*>(rho), static_cast<const float*>(ux),
                           static_cast<const float*>(uy), parity, y0, y1, rho_max, bad, st);
    return init_rows_t(h, d, static_cast<const double*>(rho), static_cast<const double*>(ux),
                       static_cast<const double*>(uy), parity, y0, y1, rho_max, bad, st);
}

cudaError_t aux_check_init(const void* rho, const void* ux, const void* uy, bool f32, long long N, double rho_max,
                           int* bad, cudaStream_t st) {
    if (f32)
        k_check_init<float><<<grid_for(N), kThreads, 0, st>>>(static_cast<const float*>(rho),
                                                               static_cast<const float*>(ux),
                                                               static_cast<const float*>(uy), N, rho_max, bad);
    else
        k_check_init<double><<<grid_for(N), kThreads, 0, st>>>(static_cast<const double*>(rho),
                                                                static_cast<const double*>(ux),
                                                                static_cast<const double*>(uy), N, rho_max, bad);
    return cudaGetLastError();
}

cudaError_t aux_fill_ghosts(const Inst& h, const Inst* d, int parity, const Notice& to, const int* word,
                            cudaStream_t st) {
    const long long M = 9ll * (4 * (h.nx + 4) + 4 * h.ny);
    if (h.prec == LBM_FP32)
        k_ghosts<float><<<grid_for(M), kThreads, 0, st>>>(d, parity, to, word);
    else
        k_ghosts<double><<<grid_for(M), kThreads, 0, st>>>(d, parity, to, word);
    return cudaGetLastError();
}

cudaError_t aux_gather_plane(const Inst& h, const Inst* d, int parity, int a, double* out, cudaStream_t st) {
    if (h.prec == LBM_FP32)
        k_gather<float><<<grid_2d(h.nx, h.ny), kThreads, 0, st>>>(d, parity, a, out);
    else
        k_gather<double><<<grid_2d(h.nx, h.ny), kThreads, 0, st>>>(d, parity, a, out);
    return cudaGetLastError();
}

template <typename O>
cudaError_t field_t(const Inst& h, const Inst* d, int parity, int field, int y0, int y1, O* out,
                    const Notice& to, cudaStream_t st) {
    const dim3 g = grid_2d(h.nx, y1 - y0);
    auto go = [&](auto k) { k<<<g, kThreads, 0, st>>>(d, parity, y0, y1, out, to); };
    const bool f32 = h.prec == LBM_FP32;
    if (field == 0) f32 ? go(k_field<float, 0, O>) : go(k_field<double, 0, O>);
    else f32 ? go(k_field<float, 3, O>) : go(k_field<double, 3, O>);
    return cudaGetLastError();
}

cudaError_t aux_field(const Inst& h, const Inst* d, int parity, int field, int y0, int y1, void* out, bool f32out,
                      const Notice& to, cudaStream_t st) {
    if (field != 0 && field != 3) return cudaErrorInvalidValue;
    if (f32out) return field_t(h, d, parity, field, y0, y1, static_cast<float*>(out), to, st);
    return field_t(h, d, parity, field, y0, y1, static_cast<double*>(out), to, st);
}

// Blocks of the flow and reduction kernels: one per tile up to what the
// device holds at once (eight blocks of 256 threads on each of 152 SMs).
constexpr int kResident = 8 * 152;
template <int NT> int flow_grid(int nx, int rows) {
    constexpr int Y = FlowTile<NT>::Y;
    const long long tiles = static_cast<long long>((nx + kFlowX - 1) / kFlowX) * ((rows + Y - 1) / Y);
    return static_cast<int>(tiles < kResident ? tiles : kResident);
}
// whether the small tiles all find an SM of their own
bool flow_small(int nx, int rows) { return flow_grid<128>(nx, rows) <= kReduceBlocks / 2; }

template <int NT, typename O>
cudaError_t flow_t(const Inst& h, const Inst* d, int parity, int y0, int y1, void* const out[4], const Notice& to,
                   cudaStream_t st) {
    auto go = [&](auto k) {
        k<<<flow_grid<NT>(h.nx, y1 - y0), NT, 0, st>>>(d, parity, y0, y1, static_cast<O*>(out[0]), static_cast<O*>(out[1]),
                                                       static_cast<O*>(out[2]), static_cast<O*>(out[3]), to);
    };
    if (h.prec == LBM_FP32) go(k_flow<NT, float, O>);
    else go(k_flow<NT, double, O>);
    return cudaGetLastError();
}
cudaError_t aux_flow(const Inst& h, const Inst* d, int parity, int y0, int y1, void* const out[4], bool f32out,
                     const Notice& to, cudaStream_t st) {
    if (flow_small(h.nx, y1 - y0))
        return f32out ? flow_t<128, float>(h, d, parity, y0, y1, out, to, st)
                      : flow_t<128, double>(h, d, parity, y0, y1, out, to, st);
    return f32out ? flow_t<256, float>(h, d, parity, y0, y1, out, to, st)
                  : flow_t<256, double>(h, d, parity, y0, y1, out, to, st);
}

cudaError_t aux_measure(const Inst& h, const Inst* d, int parity, double cxc, double cyc, double r_in,
                        double r_out, bool exact, double* partials, int rows, const Notice& to, cudaStream_t st) {
    if (rows > kResident) rows = kResident;
    const Discs D = make_discs(h.nx, h.ny, cxc, cyc, r_in, r_out);
    const int rpt = tile_rpt(h.nx, h.ny);
    const long long tiles = tile_count(h.nx, h.ny, rpt);
    const int g = static_cast<int>(tiles < rows ? tiles : rows);
    auto go = [&](auto k) { k<<<g, kLapThreads, 0, st>>>(d, parity, D, rpt, partials, to); };
    if (h.prec == LBM_FP32) exact ? go(k_measure<float, true>) : go(k_measure<float, false>);
    else exact ? go(k_measure<double, true>) : go(k_measure<double, false>);
    return cudaGetLastError();
}
bool aux_measure_again(const double (&sums)[kReduceSlots]) { return on_the_pole(sums); }

cudaError_t aux_stats(const Inst& h, const Inst* d, int parity, double* partials, int rows, const Notice& to,
                      cudaStream_t st) {
    const bool small = flow_small(h.nx, h.ny);
    const int tiles = small ? flow_grid<128>(h.nx, h.ny) : flow_grid<256>(h.nx, h.ny), g = tiles < rows ? tiles : rows;
    auto go = [&](auto k, int threads) { k<<<g, threads, 0, st>>>(d, parity, partials, to); };
    if (h.prec == LBM_FP32) small ? go(k_stats<128, float>, 128) : go(k_stats<256, float>, 256);
    else small ? go(k_stats<128, double>, 128) : go(k_stats<256, double>, 256);
    return cudaGetLastError();
}

cudaError_t aux_math_check(long long n, double lo, double hi, unsigned long long* out) {
    k_math_check<<<1024, kThreads>>>(n, lo, hi, out);
    return cudaGetLastError();
}

}  // namespace lbm
