// Register DFTs and sample conversion shared by the F-stage kernels.
#pragma once

#include <cstdint>

#include "corr_internal.h"

namespace corr {
namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// x * exp(-2 pi i a / 16) for a compile-time a in 0..7 (the roots a DFT of size <= 16 uses);
// the constants are cos and sin of multiples of pi / 8, correctly rounded to float
template <int A>
__device__ __forceinline__ float2 rot16(float2 x) {
    constexpr float kC1 = 0.92387953251128676f;   // cos(pi / 8)
    constexpr float kS1 = 0.38268343236508977f;   // sin(pi / 8)
    constexpr float kH = 0.70710678118654752f;    // cos(pi / 4)
    if constexpr (A == 0) return x;
    else if constexpr (A == 4) return make_float2(x.y, -x.x);
    else if constexpr (A == 2) return make_float2(kH * (x.x + x.y), kH * (x.y - x.x));
    else if constexpr (A == 6) return make_float2(kH * (x.y - x.x), -kH * (x.x + x.y));
    else if constexpr (A == 1) return cmul(x, make_float2(kC1, -kS1));
    else if constexpr (A == 3) return cmul(x, make_float2(kS1, -kC1));
    else if constexpr (A == 5) return cmul(x, make_float2(-kS1, -kC1));
    else return cmul(x, make_float2(-kC1, -kS1));
}

template <int M>
__host__ __device__ constexpr int bit_reverse(int r) {
    int o = 0;
    for (int b = 0; b < M; ++b) o |= ((r >> b) & 1) << (M - 1 - b);
    return o;
}

// one radix-2 butterfly level of an in-register DIT DFT: groups of SIZE, element j of a group
// combined with j + SIZE / 2 after a rotation by exp(-2 pi i j / SIZE)
template <int R, int SIZE, int J>
__device__ __forceinline__ void dit_level(float2 (&x)[R], int k0) {
    if constexpr (J < SIZE / 2) {
        const float2 u = x[k0 + J];
        const float2 t = rot16<J * (16 / SIZE)>(x[k0 + J + SIZE / 2]);
        x[k0 + J] = cadd(u, t);
        x[k0 + J + SIZE / 2] = csub(u, t);
        dit_level<R, SIZE, J + 1>(x, k0);
    }
}

template <int R, int SIZE>
__device__ __forceinline__ void dit_levels(float2 (&x)[R]) {
    if constexpr (SIZE <= R) {
#pragma unroll
        for (int k0 = 0; k0 < R; k0 += SIZE) dit_level<R, SIZE, 0>(x, k0);
        dit_levels<R, SIZE * 2>(x);
    }
}

// forward R-point DFT in registers (R = 2, 4, 8, 16): y_q = sum_r v_r exp(-2 pi i r q / R)
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&v)[R]) {
    constexpr int M = R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1;
    float2 x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[bit_reverse<M>(r)] = v[r];
    dit_levels<R, 2>(x);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[r];
}

// bytes per packed sample: 2 for complex 8-bit, 1 otherwise
template <int KIND>
__host__ __device__ constexpr int f_bps() { return KIND == CORR_F_COMPLEX8 ? 2 : 1; }

// small integers to float by the 2^23 exponent trick: a byte u (or nibble) placed in the low
// mantissa of 2^23 gives the float 2^23 + u exactly; the sign offset is flipped into u first
// (u = x + 128 for a signed byte, x + 8 for a signed nibble), then one exact subtraction
__device__ __forceinline__ float f_byte(uint32_t w, uint32_t sel, float bias) {
    return __int_as_float((int)__byte_perm(w, 0x4B000000u, sel)) - bias;
}
constexpr float kBias8 = 8388736.0f;   // 2^23 + 128
constexpr float kBias4 = 8388616.0f;   // 2^23 + 8

// one packed sample -> complex float (exact)
template <int KIND>
__device__ __forceinline__ float2 unpack1(uint32_t r) {
    if constexpr (KIND == CORR_F_COMPLEX8) {
        const uint32_t w = r ^ 0x8080u;
        return make_float2(f_byte(w, 0x7540u, kBias8), f_byte(w, 0x7541u, kBias8));
    } else if constexpr (KIND == CORR_F_COMPLEX4) {
        const uint32_t w = r ^ 0x88u;
        return make_float2(f_byte((w >> 4) & 15u, 0x7540u, kBias4), f_byte(w & 15u, 0x7540u, kBias4));
    } else {
        return make_float2(f_byte(r ^ 0x80u, 0x7540u, kBias8), 0.f);
    }
}

}  // namespace
}  // namespace corr
