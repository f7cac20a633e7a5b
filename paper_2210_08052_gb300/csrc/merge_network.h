// Steps of an in-place sorting network (Batcher's bitonic merge with the
// first step of every merge mirrored), for any number of places: every
// comparator puts the smaller value first, so places past the end need no
// values and take no part.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define MP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MP_HOST_DEVICE inline
#endif

namespace mpdp {

// step(j) for each step in order: it compares place i with place i ^ j for
// every i below i ^ j, where both are below n.  K (K + 1) / 2 steps with
// K = ceil(log2 n).  The merge's width k is 64 bits wide: in 32 bits it never
// passes 2n once n is above 2^30, and the steps would not end.
template <typename Step>
MP_HOST_DEVICE void network_steps(uint32_t n, Step step)
{
    for (uint64_t k = 2; k < 2 * static_cast<uint64_t>(n); k <<= 1)
        for (uint64_t j = k - 1; j > 0; j = j == k - 1 ? k >> 2 : j >> 1) step(static_cast<uint32_t>(j));
}

}  // namespace mpdp
