// Test driver for the words that hold rows of voltages (voltage_words.h), built by test_voltage_words.py with the
// host compiler.  Rows of T x C frames of `bytes` bytes at every address modulo 4, read word by word as the
// tensor-core gridding kernel stages them.  Output: bytes read outside the block, row bytes that came out wrong.
#include <cstdio>
#include <cstring>
#include <vector>

#include "voltage_words.h"

int main()
{
    long outside = 0, wrong = 0;
    for (int bytes = 1; bytes <= 13; ++bytes)
        for (int at = 0; at < 4; ++at) {
            const int C = 3, T = 4;
            std::vector<uint32_t> mem((T * C * bytes + 16) / 4 + 2);
            uint8_t* base = reinterpret_cast<uint8_t*>(mem.data());
            for (size_t i = 0; i < 4 * mem.size(); ++i) base[i] = (uint8_t)(i * 37 + 11);
            const uint8_t *lo = base + 4 + at, *hi = lo + (size_t)T * C * bytes;
            auto read = [&](const uint8_t* q) {
                outside += q < lo || q >= hi;
                return *q;
            };
            auto word = [&](const uint8_t* q) -> uint32_t {
                if (!epic::in_block(q, 4, lo, hi)) return epic::edge_word(q, lo, hi, read);
                uint32_t v = 0;
                for (int b = 0; b < 4; ++b) v |= (uint32_t)read(q + b) << (8 * b);
                return v;
            };
            for (int row = 0; row < T * C; ++row) {
                const uint8_t* r = lo + (size_t)row * bytes;
                const int o = (int)((uintptr_t)r & 3), nw = epic::row_words(o, bytes);
                std::vector<uint32_t> staged(nw);
                for (int j = 0; j < nw; ++j) staged[j] = word(r - o + 4 * j);
                wrong += std::memcmp(reinterpret_cast<uint8_t*>(staged.data()) + o, r, bytes) != 0;
                // shifted to a word boundary
                std::vector<uint32_t> shifted((bytes + 3) / 4);
                for (int j = 0; j < (int)shifted.size(); ++j) {
                    const uint64_t w = word(r - o + 4 * j) |
                                       (4 * j + 4 < o + bytes ? (uint64_t)word(r - o + 4 * j + 4) << 32 : 0);
                    shifted[j] = (uint32_t)(w >> (8 * o));
                }
                wrong += std::memcmp(shifted.data(), r, bytes) != 0;
            }
        }
    std::printf("%ld %ld\n", outside, wrong);
    return 0;
}
