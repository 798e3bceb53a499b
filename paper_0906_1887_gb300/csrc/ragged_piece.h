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

// The 0 to 3 bytes after the last whole word of the n_bytes at `base`, as the low bytes of a word: a thread
// reads them once, so that load_piece has no branch and its loads can be in flight together (with the
// bytes in a branch of load_piece: 75 inputs x 333 channels x 776 samples x 2 dumps 98.5 -> 102.3 us).
CORR_HOST_DEVICE uint32_t tail_word(const unsigned char* base, int64_t n_bytes) {
    uint32_t part = 0;
    for (int b = 0; b < (int)(n_bytes & 3); ++b) part |= (uint32_t)base[(n_bytes & ~(int64_t)3) + b] << (8 * b);
    return part;
}

// Bytes off .. off + 15 of the n_bytes at `base` (4-byte aligned) as four little-endian words, from the
// aligned words around them; bytes from off + n_valid on are zero.  Nothing past base + n_bytes is
// read: the last word of a buffer that is no multiple of 4 bytes is `tail` (tail_word), and so is what stands for
// the words after it, of which no byte is wanted: off + n_valid <= n_bytes, or the caller reads the bytes that
// are there only (a zero for them is one more select per word: 57 inputs x 282 channels x 158 samples,
// 4-bit, 12.4 -> 13.4 us).
CORR_HOST_DEVICE void load_piece(const unsigned char* base, int64_t off, int64_t n_bytes, int n_valid, uint32_t tail,
                                 uint32_t (&v)[4]) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(base);
    const int64_t i = off >> 2, whole = n_bytes >> 2;
    const uint32_t sh = (uint32_t)(off & 3) * 8;
    const int avail = (int)(whole - i < 5 ? whole - i : 5);   // whole words from the first on
    uint32_t x[5];
    for (int k = 0; k < 5; ++k) x[k] = k < avail ? w[i + k] : tail;
    for (int k = 0; k < 4; ++k) {
        const int left = n_valid - 4 * k;   // bytes of this word that are wanted
        v[k] = (uint32_t)((((uint64_t)x[k + 1] << 32) | x[k]) >> sh);
        if (left < 4) v[k] = left <= 0 ? 0u : v[k] & ((1u << (8 * left)) - 1u);
    }
}

}  // namespace corr
