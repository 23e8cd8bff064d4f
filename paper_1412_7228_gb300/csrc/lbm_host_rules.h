// lbm_host_rules.h -- decisions that the host takes by arithmetic alone, apart
// from the CUDA calls around them so that they can be tested without a GPU.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace lbm {

// ---- arrays that kernels reach where they lie in host memory ---------------
struct Span {
    uintptr_t at;
    size_t bytes;
};

// Whether kernels may access the array as values of `size` bytes where it
// lies: at a multiple of the size (a kernel's access to any other address
// faults), and within one mapped range, the one that its first byte is in.
// (The addresses of its two ends do not tell: with unified addressing they
// are as far apart for two ranges with unmapped pages between them.)
inline bool in_place(Span array, size_t size, Span range) {
    return array.at % size == 0 && array.at >= range.at && array.at - range.at <= range.bytes &&
           array.bytes <= range.bytes - (array.at - range.at);
}

// ---- the cluster schedule's strips ------------------------------------------
// One CTA per strip of `by` rows of at most `bx` nodes, in a cluster of up to
// kClusterCtas CTAs; the last strip at least two rows high.
constexpr int kClusterCtas = 16;
struct ClusterShape {
    int bx, by;
    constexpr int ctas(int ny) const { return (ny + by - 1) / by; }
    constexpr bool fits(int nx, int ny) const {
        return nx >= 2 && nx <= bx && ctas(ny) <= kClusterCtas && ny - (ctas(ny) - 1) * by >= 2;
    }
};
// The first of the shapes that fits the lattice and whose cluster the device
// can hold (can(k)); -1: none.  A device that cannot hold the many CTAs of a
// lattice's low strips may still hold the few of its high ones.
template <class Can> int pick_cluster(const ClusterShape* shapes, int count, int nx, int ny, Can can) {
    for (int k = 0; k < count; ++k)
        if (shapes[k].fits(nx, ny) && can(k)) return k;
    return -1;
}

// ---- the tile a context starts with -----------------------------------------
struct StartTile {
    int bx, by, threads, stages;
};
// By the nodes of n lattices, the nodes of the tiles that cover them (a tile
// reaches beyond a lattice's edge, and its ring and its loads are paid for there
// too), the rounds of tiles that the SMs take, and the rows (a tile at a lattice's
// upper or lower edge writes its ghost rows).  One-step launches from graphs, us per
// step.
//
// FP32.  One lattice: 128 x 16 from 2 M nodes on (2500 x 1200 40.0, with 32 x 16
// 44.2) and for wide ones of few rows from 0.5 M (50000 x 12 14.2, with 32 x 16 15.8;
// 40000 x 34 23.6, with 64 x 16 25.5); 64 x 16 from 1.1 M (1531 x 1117 24.6, with
// 128 x 16 25.6); below persistent 32 x 16 tiles (1000 x 900 14.7 and 16.4, 256^2 4.1 and
// 6.7).  A batch: 128 x 16 from 2 M, and for lattices that fill them as well as 32 x 16
// tiles (60 of 128^2 18.7, with 32 x 16 24.5; 15 of 256^2 17.7 and 22.8) where every other SM
// has one (10 of 128^2 7.0 and 7.6, but 8 of them 7.0 and 5.4) or nearly as well from 1 M
// (26 of 200^2 28.8 and 30.1, but 12 of 210^2 19.5 and 15.9); as 64 x 16 tiles if the lattices
// are large (4 of 512^2 18.0, with 128 x 16 19.1); also where one tile spans lattices that
// fill 32 x 16 tiles badly (60 of 70^2 11.1 and 16.0, but 100 of 96^2 28.5 and 26.8).  Else 64 x 16
// from 1.1 M where they fill those as well as 32 x 16 (300 of 64^2 44.4, with 32 x 16 50.1,
// with 128 x 16 62.0); else 32 x 16 (1000 slabs of 128 x 4: 84.5, with 128 x 16 120).
//
// FP64.  16 x 8 where they cover the lattices with fewer nodes (100 x 10000 345, with
// 32 x 8 385, with 32 x 32 396), up to three per SM (49 of 128 x 8 20.7, with 32 x 8 26.3), or
// where rounds of them end earlier (two take 1.03 times as long as one of 32 x 8; 400^2
// in 9 and 5 rounds: 55.9 and 60.9; 512^2 in 14 and 7: 85.4 and 84.3; 600^2 114.8 and 118.9),
// unless a batch's lattices have few rows (195 of 128 x 8, in 11 and 6: 106.7 and 94.2); 32 x 32
// from 0.9 M where their rows are filled (1024^2 308, with 32 x 8 315, but 2000 slabs of
// 128 x 4 1350 and 623); else 32 x 8.
inline StartTile start_tile(bool fp64, int n, const int* nx, const int* ny) {
    long long N = 0, columns = 0;
    int widest = 0;
    for (int i = 0; i < n; ++i) {
        N += static_cast<long long>(nx[i]) * ny[i];
        columns += nx[i];
        if (nx[i] > widest) widest = nx[i];
    }
    const double nodes = static_cast<double>(N), rows = nodes / static_cast<double>(columns);   // mean over the columns
    auto covered = [&](int bx, int by) {
        double sum = 0.0;
        for (int i = 0; i < n; ++i)
            sum += static_cast<double>((nx[i] + bx - 1) / bx * bx) * static_cast<double>((ny[i] + by - 1) / by * by);
        return sum;
    };
    constexpr int kSms = 152;
    if (fp64) {
        const double c8 = covered(32, 8), c16 = covered(16, 8);
        if (c16 <= 0.95 * c8 || c16 <= 3.0 * kSms * (16 * 8)) return {16, 8, 128, 1};
        if (N >= 900000 && covered(32, 32) <= 1.03125 * c8) return {32, 32, 256, 1};
        auto rounds = [&](double c, int size) { return static_cast<double>(static_cast<long long>((c / size + kSms - 1) / kSms)); };
        if ((n == 1 || rows >= 24.0) && 1.03 * rounds(c16, 16 * 8) < 2.0 * rounds(c8, 32 * 8)) return {16, 8, 128, 1};
        return {32, 8, 256, 1};
    }
    const StartTile wide = {128, 16, 512, 1}, mid = {64, 16, 256, 1}, narrow = {32, 16, 256, 2};
    if (N >= 2000000) return wide;
    if (n == 1) {
        if (N >= 500000 && rows < 64.0) return wide;
        return N >= 1100000 ? mid : narrow;
    }
    const double cw = covered(128, 16), cn = covered(32, 16);
    if (rows >= 32.0) {
        if (cw >= 0.5 * kSms * (128 * 16) && cw <= (N >= 1000000 ? 1.15 : 1.05) * cn) return N / n >= 200000 ? mid : wide;
        if (N >= 270000 && widest <= 128 && cw <= 1.34 * cn && cn >= 1.1 * nodes) return wide;
    }
    return N >= 1100000 && rows >= 32.0 && covered(64, 16) <= 1.01 * cn ? mid : narrow;
}

}  // namespace lbm
