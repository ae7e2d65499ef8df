// Comparison of 32-bit counts that may wrap around.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define MLD_HOST_DEVICE __host__ __device__
#else
#define MLD_HOST_DEVICE
#endif

namespace mld {

// Whether a count that only goes up has reached `target`, both modulo 2^32 and
// less than 2^31 apart.
MLD_HOST_DEVICE inline bool count_reached(uint32_t now, uint32_t target) {
    return static_cast<int32_t>(now - target) >= 0;
}

}  // namespace mld
