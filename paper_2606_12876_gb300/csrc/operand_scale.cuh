// Power-of-two scaling of codebooks into fp16's range for the tensor-core kernels that sum the
// codewords of a group and round the sum once to fp16. Internal; not part of the ABI.
#pragma once

#include "aq_internal.cuh"

namespace aq {

__device__ __forceinline__ uint32_t f16x2(float2 v) {   // {lo, hi} -> packed fp16 pair, RN
    uint32_t h;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(v.y), "f"(v.x));
    return h;
}

// fp16 range for any input (R9). The MMA operands are fp16; bf16 activations and bf16
// codebooks can hold values far outside fp16's range (and fp16 books' sums can exceed it).
// Both are therefore scaled by powers of two, which is exact: each token row of bf16
// activations by 2^-e_t so that its largest |x| lies in [2^14, 2^15) (bf16_rows_to_f16_kernel),
// and the codebooks by 2^-f so that the largest possible |sum of m codewords| (the sum over
// the books of their largest |entry|) lies below 2^15 (for bf16 books also at least 2^14, so
// that small weights do not fall into fp16's subnormal range; fp16 books are only scaled down,
// and a single fp16 book not at all). The epilogue multiplies by 2^e_t and by s 2^f: the scaled sums
// stay below about 2^46, so the order that overflows only where y does is s 2^f first for e_t > 0 and
// 2^e_t first otherwise. (Always 2^e_t first, activations of 2^112 and weights of 2^-4, scaled by 2^18,
// gave infinity for y of about 2^112.) Where nothing was out of range the result is bit-identical to the
// unscaled computation.

// Largest finite |entry| of a codeword of eight 16-bit values, as the bits of a non-negative float
// (monotonic in the value, so unsigned maxima of them are maxima of the values). Infinities and NaN stay
// what they are at any scale; counted here, one infinite entry would scale every finite one to zero.
template <int BDT>
__device__ __forceinline__ unsigned int codeword_max_bits(const uint4& c) {
    float f[8];
    unpack8<BDT>(c, f);
    float mx = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) mx = fmaxf(mx, fabsf(f[e]) < INFINITY ? fabsf(f[e]) : 0.0f);
    return __float_as_uint(mx);
}

// f of the codebooks of prefix m from the per-book largest |entry| (float bits).
template <int BDT>
__device__ __forceinline__ int book_exponent(const unsigned int* wmax, int m) {
    if (BDT == AQ_F16 && m == 1) return 0;   // one fp16 codeword is an fp16 value already
    float tot = 0.0f;
    for (int k = 0; k < m; ++k) tot += __uint_as_float(wmax[k]);
    if (!(tot > 0.0f)) return 0;             // no finite entry but zeros
    int f = exponent_of(fminf(tot, 3.0e38f)) - 14;
    if (BDT == AQ_F16 && f < 0) f = 0;
    return max(-126, f);                     // (at most 113; the smallest bf16 value is 2^-133)
}

// A codeword times sc (a power of two), back in its own type.
template <int BDT>
__device__ __forceinline__ uint4 scale_codeword(const uint4& c, float sc) {
    float f[8];
    unpack8<BDT>(c, f);
    uint16_t h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) h[e] = f32_to_bits<BDT>(f[e] * sc);
    return make_uint4(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16),
                      h[4] | ((uint32_t)h[5] << 16), h[6] | ((uint32_t)h[7] << 16));
}

}  // namespace aq
