// Phases of the two mbarriers on which a kernel commits the MMAs of its tiles, one
// barrier per accumulator, the accumulators in turn. Plain C++: the host compiles it
// too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CS_HD __host__ __device__
#else
#define CS_HD
#endif

struct MmaPhase {
    uint32_t bar, parity;
};

// Barrier and phase parity of tile number `tile` (from 0 over the CTA's life).
CS_HD constexpr MmaPhase mma_phase(uint32_t tile) { return {tile & 1u, (tile >> 1) & 1u}; }

// The phase that ends when the MMAs of all `issued` tiles have: a commit covers
// every MMA that its thread issued before it, so the last tile's. (Its parity tells
// it from the phase before only once tile issued - 3 on the same barrier is done,
// which the issuer makes sure of: it issues a tile when the second one before it has
// been waited for.) False: nothing was issued.
CS_HD constexpr bool mma_last(uint32_t issued, MmaPhase& p) {
    if (issued == 0) return false;
    p = mma_phase(issued - 1u);
    return true;
}
