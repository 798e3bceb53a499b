// Exact conversion of packed 4/8-bit complex samples to fp16, shared by the fused
// tensor-core kernel's converter warps and the standalone unpack kernel.
//
// fp16(1024 + u) has the bit pattern 0x6400 | u for 0 <= u < 1024.  For two samples taken
// from byte lane `sel` of words a and b, (r & 0x00FF00FF) ^ flip both inserts the 0x64
// exponent bytes and turns each two's-complement byte (or nibble) into u = x + offset; one
// half2 subtraction of 1024 + offset then leaves x exactly.
#pragma once

#include <cuda_fp16.h>
#include <cstdint>

namespace corr {
namespace conv {

__device__ __forceinline__ uint32_t pair_to_half2(uint32_t a, uint32_t b, uint32_t sel, uint32_t flip, __half2 bias) {
    uint32_t r = (__byte_perm(a, b, sel) & 0x00FF00FFu) ^ flip;
    __half2 h = __hsub2(*reinterpret_cast<__half2*>(&r), bias);
    return *reinterpret_cast<uint32_t*>(&h);
}

// byte-permute selector placing byte k of a in byte 0 and byte k of b in byte 2
__device__ __forceinline__ uint32_t lane_selector(int k) {
    return (uint32_t)(k | (k << 4) | ((k + 4) << 8) | ((k + 4) << 12));
}

// 8-bit samples: flip the sign bit of each byte, bias 1024 + 128
__device__ __forceinline__ __half2 bias8() {
    return __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));   // 1152
}
constexpr uint32_t kFlip8 = 0x64806480u;

// 4-bit samples (one nibble per byte lane after masking): flip bit 3, bias 1024 + 8
__device__ __forceinline__ __half2 bias4() {
    return __halves2half2(__ushort_as_half(0x6408), __ushort_as_half(0x6408));   // 1032
}
constexpr uint32_t kFlip4 = 0x64086408u;

// 4-bit samples to e4m3 by table.  prmt picks a byte of an 8-byte table per selector nibble; a set
// top bit of the nibble gives the byte's sign instead, 0x00 for tables of magnitudes.  With the
// two's complement nibble n as selector, table kMag picks |n| for n >= 0 and 0 for n < 0; with the
// top bit flipped, table kNeg picks |n| for n < 0 and 0 for n >= 0.  Two lookups convert four
// nibbles; the signs are the nibbles' top bits.  17 integer instructions per 8 values, against 21 with
// four hardware conversions from fp16 among them (64 inputs x 768 channels x 1000 samples x 4 dumps
// 111 -> 97 us, 128 x 512 x 2048 81 -> 71).
constexpr uint32_t kMagLo = 0x44403800u, kMagHi = 0x4E4C4A48u;   // e4m3 of 0 .. 7
constexpr uint32_t kNegLo = 0x4A4C4E50u, kNegHi = 0x38404448u;   // e4m3 of 8, 7 .. 1: |n - 16| for n = 8 .. 15

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// u: four samples (re nibble high, im nibble low) of one input -> their re and im values as e4m3 bytes
__device__ __forceinline__ void e4m3_of_nibbles(uint32_t u, uint32_t& re, uint32_t& im) {
    const uint32_t f = u ^ 0x88888888u;
    const uint32_t m01 = prmt(kMagLo, kMagHi, u) | prmt(kNegLo, kNegHi, f);   // |im0|, |re0|, |im1|, |re1|
    const uint32_t m23 = prmt(kMagLo, kMagHi, u >> 16) | prmt(kNegLo, kNegHi, f >> 16);
    re = prmt(m01, m23, 0x7531u) | (u & 0x80808080u);
    im = prmt(m01, m23, 0x6420u) | ((u << 4) & 0x80808080u);
}

// byte k of four words, one per byte; sel = gather_selector(k)
__host__ __device__ constexpr uint32_t gather_selector(int k) { return (uint32_t)k | ((uint32_t)(4 + k) << 4); }
__device__ __forceinline__ uint32_t gather4(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t sel) {
    return prmt(prmt(w0, w1, sel), prmt(w2, w3, sel), 0x5410u);
}

}  // namespace conv
}  // namespace corr
