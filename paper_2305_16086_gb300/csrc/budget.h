// Device memory a traversal may take for what grows with the graph times the
// launch: one rule for the windowed loop's ping-pong buffers and the resident
// traversal's node marks. Plain C++.
#pragma once

#include <algorithm>
#include <cstddef>

namespace sc {

// at most 4 GB, and an eighth of what is free
inline double traversal_budget(size_t free_bytes) {
    return std::min(4.0 * (1ull << 30), 0.125 * static_cast<double>(free_bytes));
}

// CTAs of the resident class whose adjacency lies in global memory for `sources` sources on `sms` SMs, `bytes`
// of device memory each: one per SM, or none when the budget does not hold them (`held` bytes are allocated)
inline int global_class_ctas(size_t bytes, size_t sources, int sms, size_t held, size_t free_bytes) {
    const size_t ctas = std::min(sources, static_cast<size_t>(std::max(sms, 1)));
    const size_t need = bytes * ctas;
    return need <= held || static_cast<double>(need) <= traversal_budget(free_bytes + held) ? static_cast<int>(ctas) : 0;
}

}  // namespace sc
