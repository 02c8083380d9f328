// Eight-byte words of a row of labels at any alignment.  Plain C++ but for the
// qualifiers, so that a host test can count the bytes it reads.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define VESIS_HD __host__ __device__ __forceinline__
#else
#define VESIS_HD inline
#endif

namespace vesis {

// Cells k0 - 8 .. k0 - 1, k0 .. k0 + 7 and k0 + 8 .. k0 + 15 (lo, mid, hi) of the
// row of nz one-byte cells that starts `at` bytes into an array of `size` (below
// 2^31) bytes at `base`; k0 a multiple of 8 below nz, cells past the row's ends
// zero.  word(p) loads the aligned word at p, byte(p) one byte.  The up to four
// aligned words that hold cells of the row are shifted into place.  Words of a
// row within 8 bytes of the array's ends could stick out of it: there the cells
// are read one by one.
template <class Word, class Byte>
VESIS_HD void row_words(uintptr_t base, unsigned at, int k0, int nz, unsigned size, Word word,
                        Byte byte, uint64_t &lo, uint64_t &mid, uint64_t &hi)
{
    const uintptr_t row = base + at;
    if (at < 8u || at + (unsigned)nz + 8u > size) {
        uint64_t v[3] = {0u, 0u, 0u};
        for (int c = k0 < 8 ? 8 - k0 : 0; c < 24 && k0 + c - 8 < nz; ++c) {
            const uint64_t b = (uint64_t)byte(row + (uintptr_t)(k0 + c - 8)) << (8 * (c & 7));
            if (c < 8) v[0] |= b;
            else if (c < 16) v[1] |= b;
            else v[2] |= b;
        }
        lo = v[0];
        mid = v[1];
        hi = v[2];
        return;
    }
    const int m = (int)((row + (uintptr_t)k0) & 7u);
    const uintptr_t p = row + (uintptr_t)k0 - (uintptr_t)m;      // aligned
    uint64_t v[4];                       // aligned words from cell k0 - 8 - m on
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int z = k0 - m + 8 * (e - 1);
        v[e] = z + 8 > 0 && z < nz ? word(p + (uintptr_t)(8 * e) - 8u) : 0u;
    }
    if (m) {
#pragma unroll
        for (int e = 0; e < 3; ++e) v[e] = (v[e] >> (8 * m)) | (v[e + 1] << (64 - 8 * m));
    }
    const auto upto = [](int c) {        // the first c bytes of a word
        return c >= 8 ? ~(uint64_t)0 : c <= 0 ? 0u : ((uint64_t)1 << (8 * c)) - 1u;
    };
    lo = k0 >= 8 ? v[0] : 0u;
    mid = v[1] & upto(nz - k0);
    hi = v[2] & upto(nz - k0 - 8);
}

}  // namespace vesis
