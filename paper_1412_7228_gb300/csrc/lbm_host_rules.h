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

}  // namespace lbm
