// lbm_reduce.cuh -- FP64 sums over a lattice or a field in one launch: the
// per-block reduction, the last block's sum of the blocks' partial sums, and
// the disc tests of the Laplace sampling.  Shared by lbm_aux.cu and
// lbm_static.cu.
//
// GB300's FP64 pipe (two thread operations per clock and SM) bounds all of
// these, so the code around the sums spends as few FP64 instructions as it
// can: an FP64 instruction of one warp holds the pipe for 16 to 19 clocks
// however many of its lanes carry data, and conversions to and from FP64 do
// as well.
#pragma once

#include <cmath>

#include "lbm_internal.cuh"

namespace lbm {
namespace {


// Sums of eight values over a warp.  A shuffle tree per value costs 8 x 5
// FP64 additions per warp; here each exchange halves the values a lane
// still carries (4 + 2 + 1 additions for the eight values, then two more),
// nine in all.  The sum of slot k ends in the four lanes 4k .. 4k + 3.
__device__ __forceinline__ double warp_sum8(const double (&v)[8]) {
    const int lane = threadIdx.x & 31;
    double a[4], b[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool up = lane & 16;   // this half keeps slots 4..7
        const double keep = up ? v[k + 4] : v[k], give = up ? v[k] : v[k + 4];
        a[k] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool up = lane & 8;
        const double keep = up ? a[k + 2] : a[k], give = up ? a[k] : a[k + 2];
        b[k] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    const bool up = lane & 4;
    double x = (up ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    return x + __shfl_xor_sync(0xffffffffu, x, 1);
}

// The blocks' sums (slot max_slot: maximum; -1: none) of v over all threads
// of the grid, written by the last block to finish: every block stores its
// eight partial sums and draws a ticket; the block that draws the last one
// adds the partial sums in an order fixed by the grid alone, so the result
// does not depend on which block that is.  Returns true in threads 0..7 of
// the last block only, with slot threadIdx.x in *total; *ticket is back at
// zero for the next launch on the stream.  vmax: the maximum's candidate of
// this thread when max_slot >= 0 (its own v entry is ignored).
//
// The former second launch (one warp adding 304 rows one after another)
// took 45 us by itself; here the last block's groups of 8 threads take the
// rows in turn.
template <int NT>
__device__ __forceinline__ bool grid_sum8(const double (&v)[8], int max_slot, double vmax, double* partials,
                                          unsigned* ticket, double* total) {
    constexpr int kWarps = NT / 32, kGroups = NT / 8;
    __shared__ double red[kWarps][8];
    __shared__ unsigned s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double x = warp_sum8(v);
    if ((lane & 3) == 0) red[warp][lane >> 2] = x;
    if (max_slot >= 0) {
        double m = vmax;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        __syncwarp();
        if (lane == 0) red[warp][max_slot] = m;
    }
    __syncthreads();
    auto add = [&](double a, double b, int slot) { return slot == max_slot ? fmax(a, b) : a + b; };
    if (tid < 8) {
        double s = red[0][tid];
        for (int w = 1; w < kWarps; ++w) s = add(s, red[w][tid], tid);
        partials[blockIdx.x * 8 + tid] = s;
        __threadfence();   // before the ticket: whoever draws the last one sees this block's row
    }
    __syncwarp();          // threads 0..7 are all of the writers, in warp 0
    if (tid == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    const int slot = tid & 7, group = tid >> 3, n = static_cast<int>(gridDim.x);
    double s = slot == max_slot ? -INFINITY : 0.0;
    for (int b = group; b < n; b += kGroups) s = add(s, __ldcg(partials + b * 8 + slot), slot);
    s = add(s, __shfl_xor_sync(0xffffffffu, s, 8), slot);
    s = add(s, __shfl_xor_sync(0xffffffffu, s, 16), slot);
    __syncthreads();       // red is read no more
    if (lane < 8) red[warp][lane] = s;
    __syncthreads();
    if (tid == 0) *ticket = 0;
    if (tid >= 8) return false;
    double t = red[0][tid];
    for (int w = 1; w < kWarps; ++w) t = add(t, red[w][tid], tid);
    *total = t;
    return true;
}

// The Laplace discs around (cx, cy), prepared on the host: a node at
// distance d (periodic minimum image) is inside for d <= r_in and outside
// for d >= r_out, tested on d^2 against in2, the largest number whose
// correctly rounded square root is <= r_in, and out2, the smallest whose
// root is >= r_out.  Square roots are monotone, so the tests decide as
// those on d = sqrt(d^2) do, without the root.  A centre that is not finite
// puts no node in either (every d is NaN).
struct Discs {
    double cx, cy, inv_nx, inv_ny;
    long long in2, out2;   // bit patterns: d^2 >= 0, and such doubles order as their patterns
};
inline Discs make_discs(int nx, int ny, double cx, double cy, double r_in, double r_out) {
    Discs D;
    D.cx = cx;
    D.cy = cy;
    D.inv_nx = 1.0 / nx;
    D.inv_ny = 1.0 / ny;
    double a = r_in * r_in;
    while (std::sqrt(a) > r_in) a = std::nextafter(a, 0.0);
    while (std::sqrt(std::nextafter(a, INFINITY)) <= r_in && a < INFINITY) a = std::nextafter(a, INFINITY);
    double b = r_out * r_out;
    while (std::sqrt(b) < r_out) b = std::nextafter(b, INFINITY);
    while (b > 0.0 && std::sqrt(std::nextafter(b, 0.0)) >= r_out) b = std::nextafter(b, 0.0);
    if (!std::isfinite(cx) || !std::isfinite(cy)) {
        D.cx = D.cy = 0.0;
        D.in2 = -1;                        // no d^2 is below it
        D.out2 = 0x7fffffffffffffffll;     // and none above this
        return D;
    }
    auto bits = [](double v) {
        long long i;
        static_assert(sizeof i == sizeof v, "64-bit patterns");
        __builtin_memcpy(&i, &v, sizeof i);
        return i;
    };
    D.in2 = bits(a);
    D.out2 = bits(b);
    return D;
}
// Distance along one axis from the centre, minimum image, squared.  The
// multiplication by 1/n stands for a division: where the two round apart, v
// is half a period from the centre on either side, and the square is the same.
__device__ __forceinline__ double axis2(int v, double c, int n, double inv_n) {
    double d = v - c;
    d -= n * rint(d * inv_n);
    return d * d;
}

// num / den rounded like the division up to the last bit's ties: Newton's
// reciprocal (Fast<double>::rcp), then one residual step (Markstein, IBM J.
// Res. Dev. 34, 1990).  Six FP64 instructions.  NaN where den is zero or not
// finite or the quotient is infinite.
__device__ __forceinline__ double quotient(double num, double inv_den, double den) {
    const double q = num * inv_den;
    return fma(fma(-q, den, num), inv_den, q);
}
// Where that is no number, or the reciprocal leaves the normal range (den
// zero, denormal, from 2^1022 on or not finite): num and den scaled by a power
// of two first, and the product with the reciprocal's estimate (infinite or
// zero then) where the quotient still is none.  The tests are integer ones, and
// calling the division instead would cost the kernels registers (48 -> 56).
__device__ __forceinline__ bool not_a_number(double v) { return (__double2hiint(v) & 0x7fffffff) > 0x7ff00000; }
__device__ __forceinline__ double quotient_any(double num, double inv_den, double den) {
    double r = quotient(num, inv_den, den);
    if ((static_cast<unsigned>(__double2hiint(den)) << 1) - (1u << 21) >= 2044u << 21) {
        const double scale = (__double2hiint(den) & 0x7fffffff) < 0x3ff00000 ? 0x1p200 : 0x1p-200;
        num *= scale;
        den *= scale;
        r = quotient(num, Fast<double>::rcp(den), den);
    }
    return not_a_number(r) ? num * Fast<double>::estimate(den) : r;
}

// The pressure law with its constants folded, p = rho [K R T h(rho) - K a rho]
// (h = num / q^3 for Carnahan-Starling), and psi = W / sqrt(W D) with Eq.
// 10's radicand (2/G)(p - rho/3) = W / D: 16 (with the sum) and 17 FP64
// instructions.  On its pole the pressure is infinite, which quotient does not
// give; EXACT: by the division.
struct LawFp64 {
    int eos;
    double b, c1, c2, c3;   // p: K R T, K a (K a alpha), 0; psi: those and 1/3, times 2/G
    __device__ __forceinline__ LawFp64(const Phys<double>& P, bool psi) {
        const double s = psi ? P.two_over_G : 1.0;
        eos = P.eos;
        b = P.eos == LBM_EOS_CS ? P.b4 : P.b;
        c1 = s * (P.K * P.RT);
        c2 = s * (P.K * (P.eos == LBM_EOS_PR ? P.aalpha : P.a));
        c3 = psi ? s * (1.0 / 3.0) : 0.0;
    }
    // p / rho
    template <bool EXACT> __device__ __forceinline__ double pressure_over_rho(double rho) const {
        const double n = b * rho, q = 1.0 - n;
        if (eos == LBM_EOS_CS) return c1 * div<EXACT>(fma(n, fma(n, q, 1.0), 1.0), q * q * q) - c2 * rho;
        if (eos == LBM_EOS_VDW) return div<EXACT>(c1, q) - c2 * rho;
        return div<EXACT>(c1, q) - div<EXACT>(c2 * rho, fma(n, 2.0 - n, 1.0));
    }
    __device__ __forceinline__ double psi(double rho) const {
        const double n = b * rho, q = 1.0 - n;
        if (eos == LBM_EOS_CS) {
            const double q3 = q * q * q;
            return psi_fold_fp64(rho * fma(-fma(c2, rho, c3), q3, c1 * fma(n, fma(n, q, 1.0), 1.0)), q3);
        }
        if (eos == LBM_EOS_VDW) return psi_fold_fp64(rho * fma(-fma(c2, rho, c3), q, c1), q);
        const double e = fma(n, 2.0 - n, 1.0);
        return psi_fold_fp64(rho * fma(-fma(c2, rho, c3 * e), q, c1 * e), q * e);
    }
    template <bool EXACT> static __device__ __forceinline__ double div(double num, double den) {
        return EXACT ? num / den : quotient(num, Fast<double>::rcp(den), den);
    }
};

// Laplace sums of one thread: {sum rho, sum p_in, sum rho_in, n_in,
// sum p_out, sum rho_out, n_out, 0}; p = p_EOS(rho).  A node's density is
// added once: to the disc it belongs to, or to `rest` when it belongs to
// neither (taken off it when it belongs to both).
template <bool EXACT> struct LaplaceSums {
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0}, rest = 0.0;
    int n_in = 0, n_out = 0;
    __device__ __forceinline__ void add(const LawFp64& p_eos, const Discs& D, double r, double d2) {
        const long long b = __double_as_longlong(d2);
        const bool in = b <= D.in2, out = b >= D.out2;
        if (in == out) rest += in ? -r : r;
        if (!in && !out) return;
        const double p = p_eos.template pressure_over_rho<EXACT>(r);   // its product with rho goes into the sum
        if (in) {
            v[1] = fma(r, p, v[1]);
            v[2] += r;
            ++n_in;
        }
        if (out) {
            v[4] = fma(r, p, v[4]);
            v[5] += r;
            ++n_out;
        }
    }
    __device__ __forceinline__ void close() {
        v[0] = (v[2] + v[5]) + rest;
        v[3] = n_in;
        v[6] = n_out;
    }
};

// Tiles of the Laplace sums: kTileX columns by kTileRows * rpt rows, a
// thread taking rpt nodes of one column.  Blocks of four warps, one per SM
// quarter: the FP64 pipe takes 64 clocks per warp instruction of a quarter, so
// more warps on an SM only lengthen a small lattice's chain (64^2: 256
// threads per block 11.0 us on the device, 128 threads 8.3).
constexpr int kLapThreads = 128, kTileX = 64, kTileRows = kLapThreads / kTileX, kMaxRpt = 16;
inline long long tile_count(int nx, int ny, int rpt) {
    return static_cast<long long>((nx + kTileX - 1) / kTileX) * ((ny + rpt * kTileRows - 1) / (rpt * kTileRows));
}
// Rows per thread: the cheapest of 1 .. kMaxRpt in FP64 instructions of the
// busiest SM, about 23 per node and 13 per thread and tile (its distances and
// its block's reduction).
inline int tile_rpt(int nx, int ny) {
    int best = 1;
    long long least = 0;
    for (int rpt = 1; rpt <= kMaxRpt; rpt *= 2) {
        const long long cost = (tile_count(nx, ny, rpt) + 151) / 152 * (23 * rpt + 13);
        if (rpt == 1 || cost < least) {
            least = cost;
            best = rpt;
        }
    }
    return best;
}
// Whether the sums have to be formed again, by the divisions: a pressure that is
// no number over densities that are (one of them on the law's pole).
inline bool on_the_pole(const double (&s)[8]) { return std::isfinite(s[0]) && (std::isnan(s[1]) || std::isnan(s[4])); }

// The sums over the tiles of this block; rho_at(x, y) gives a node's density.
// A tile's squared distances along x and y are formed once, in shared memory,
// while the first densities arrive.
struct AxisTable {
    double x[kTileX], y[kTileRows * kMaxRpt];
};
template <bool EXACT, typename F>
__device__ __forceinline__ void laplace_tiles(LaplaceSums<EXACT>& L, const LawFp64& p_eos, const Discs& D, int nx, int ny,
                                              int rpt, AxisTable& A, F rho_at) {
    const int rows = kTileRows * rpt, t = threadIdx.x, tx = t % kTileX, ty = t / kTileX;
    const int tiles_x = (nx + kTileX - 1) / kTileX, tiles = tiles_x * ((ny + rows - 1) / rows);
    for (int k = blockIdx.x; k < tiles; k += gridDim.x) {
        const int row = k / tiles_x, x0 = (k - row * tiles_x) * kTileX, x = x0 + tx, y0 = row * rows;
        const double first = x < nx && y0 + ty < ny ? rho_at(x, y0 + ty) : 0.0;
        if (k != static_cast<int>(blockIdx.x)) __syncthreads();   // the tile before is done with the table
        for (int e = t; e < kTileX + rows; e += kLapThreads) {
            const bool along_x = e < kTileX;
            const double d = axis2(along_x ? x0 + e : y0 + e - kTileX, along_x ? D.cx : D.cy, along_x ? nx : ny,
                                   along_x ? D.inv_nx : D.inv_ny);
            (along_x ? A.x[e] : A.y[e - kTileX]) = d;
        }
        __syncthreads();
        if (x >= nx) continue;
        const double dx2 = A.x[tx];
        for (int j = ty; j < rows && y0 + j < ny; j += kTileRows)
            L.add(p_eos, D, j == ty ? first : rho_at(x, y0 + j), dx2 + A.y[j]);
    }
    L.close();
}

}  // namespace
}  // namespace lbm
