// Sums over the lanes of a warp of several values at once.
#pragma once

namespace hm {

// The sums over the warp of NV values per lane (NV a power of two): halving exchanges, then
// butterflies -- every value adds its lanes in the order of a plain xor butterfly from 16
// down, so the sum is the same bit for bit.  Returns the index of the value whose sum this
// lane holds in v[0].
template <int NV, typename T>
__device__ __forceinline__ int warp_sums(T (&v)[NV], int lane) {
    int k = 0;
#pragma unroll
    for (int h = NV / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const T mine = up ? v[j + h] : v[j], other = up ? v[j] : v[j + h];
            v[j] = mine + __shfl_xor_sync(0xffffffffu, other, o);
        }
        if (up) k += h;
    }
#pragma unroll
    for (int o = 16 / NV; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return k;
}

}  // namespace hm
