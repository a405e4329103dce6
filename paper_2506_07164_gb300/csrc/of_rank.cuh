// Order of candidates: the unique 96-bit rank word R = (key ^ 2^63) << 32 |
// ~((y << 16) | x), larger = better (Harris key descending, then y, then x
// ascending), and a 12-bit code of the key that is monotone in it.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ofk {

__device__ __forceinline__ bool rank_less(uint64_t ah, uint32_t al, uint64_t bh, uint32_t bl) {
    return ah < bh || (ah == bh && al < bl);
}

// f(x) for 0 <= x < 2^63: 0 for x = 0, else 32 * bitlength(x) + the 5 bits
// after the leading one -- non-decreasing in x, at most 2047.
__device__ __forceinline__ uint32_t mag_code(uint64_t x) {
    if (x == 0ull) return 0u;
    const int L = 64 - __clzll((long long)x);
    return 32u * (uint32_t)L + (uint32_t)((x << (64 - L)) >> 58 & 31ull);
}

// Code of the order-preserving key u = key ^ 2^63, non-decreasing in key:
// keys >= 0 map to 2048 + f(key), keys < 0 to 2047 - f(-key - 1).
__device__ __forceinline__ uint32_t key_code(uint64_t u) {
    return (u >> 63) ? 2048u + mag_code(u & 0x7FFFFFFFFFFFFFFFull) : 2047u - mag_code(u ^ 0x7FFFFFFFFFFFFFFFull);
}

}  // namespace ofk
