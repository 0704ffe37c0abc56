// The aligned 4-byte words that hold a row of voltages, read without touching what lies around the caller's block.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace epic {

// words that hold the `bytes` bytes of a row which begins `o` bytes into its first word
__host__ __device__ inline int row_words(int o, int bytes) { return (o + bytes + 3) >> 2; }

// n bytes from w lie in the block [lo, hi)
__host__ __device__ inline bool in_block(const uint8_t* w, size_t n, const uint8_t* lo, const uint8_t* hi)
{
    return w >= lo && w + n <= hi;
}

// A word at an end of the block: its bytes in [lo, hi) by byte(address), zeros for the others.
template <class Byte>
__host__ __device__ inline uint32_t edge_word(const uint8_t* w, const uint8_t* lo, const uint8_t* hi, Byte&& byte)
{
    uint32_t v = 0;
    for (int b = 0; b < 4; ++b)
        if (w + b >= lo && w + b < hi) v |= (uint32_t)byte(w + b) << (8 * b);
    return v;
}

}  // namespace epic
