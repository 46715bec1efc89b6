// grid_limits.h - what the persistent grid solvers can address, in plain
// integers (no CUDA, so that it is tested on the host).
#pragma once

#include <stdint.h>

namespace gk {

// Whether 32-bit byte offsets reach every entry of an ELL matrix of K entries
// a row and the given stride: of its values (value_bytes each) and of its
// int32 columns, which take the larger offsets beside 16-bit values.  A chunk
// of 8 entries past a row's last is formed, not read, so K counts 8 more.
inline bool grid_offsets_fit(int64_t K, int64_t stride, int64_t value_bytes) {
    const uint64_t entry = (uint64_t)(value_bytes > 4 ? value_bytes : 4);
    return ((uint64_t)K + 8) * (uint64_t)stride <= ((1ull << 32) - 1) / entry;
}

}  // namespace gk
