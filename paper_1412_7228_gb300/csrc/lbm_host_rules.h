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
// faults).
inline bool in_place(Span array, size_t size) { return array.at % size == 0; }

}  // namespace lbm
