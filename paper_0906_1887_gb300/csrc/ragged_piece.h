// 16 bytes of packed samples from any byte offset, for rows that are no 16-byte multiples.  Plain
// C++ on either side of the compiler, so that the reads can be checked on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CORR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define CORR_HOST_DEVICE inline
#endif

namespace corr {

// Bytes off .. off + 15 of the n_bytes at `base` (4-byte aligned) as four little-endian words, from the
// aligned words around them; bytes from off + n_valid on are zero.  Nothing past base + n_bytes is
// read: the words there count as zero, and the last word of a buffer that is no multiple of 4 bytes is
// put together byte by byte (in the one or two pieces that reach it).
CORR_HOST_DEVICE void load_piece(const unsigned char* base, int64_t off, int64_t n_bytes, int n_valid, uint32_t (&v)[4]) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(base);
    const int64_t i = off >> 2, whole = n_bytes >> 2;
    const uint32_t sh = (uint32_t)(off & 3) * 8;
    uint32_t x[5];
    if (i + 5 <= whole) {
        for (int k = 0; k < 5; ++k) x[k] = w[i + k];
    } else {
        for (int k = 0; k < 5; ++k) {
            x[k] = 0u;
            if (i + k < whole) x[k] = w[i + k];
            else if (i + k == whole)
                for (int b = 0; b < (int)(n_bytes & 3); ++b) x[k] |= (uint32_t)base[4 * whole + b] << (8 * b);
        }
    }
    for (int k = 0; k < 4; ++k) {
        const int left = n_valid - 4 * k;   // bytes of this word that are wanted
        v[k] = (uint32_t)((((uint64_t)x[k + 1] << 32) | x[k]) >> sh);
        if (left < 4) v[k] = left <= 0 ? 0u : v[k] & ((1u << (8 * left)) - 1u);
    }
}

}  // namespace corr
