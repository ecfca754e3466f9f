// The neighbour lists of the pair kernel for more than two species
// (k_pair_multi.cuh): one list per particle, read by L lanes together.
#pragma once

#include "launch.h"

namespace tdpd {

// Entry e of particle i's list, L lanes per particle: the particles of a warp's
// 32 / L lane groups are interleaved in blocks of 32 entries, L of each, so that
// the L lanes of a particle read consecutive entries and a warp reads whole
// 128-byte lines (capb = capacity / L blocks).
__host__ __device__ __forceinline__ size_t striped_row(int i, int L, int capb)
{
    const int p1 = 32 / L;
    return (size_t)(i / p1) * capb * 32 + (i % p1) * L;
}
__host__ __device__ __forceinline__ int striped_off(int e, int L) { return (e / L) * 32 + e % L; }

}  // namespace tdpd
