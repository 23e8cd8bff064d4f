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

}  // namespace lbm
