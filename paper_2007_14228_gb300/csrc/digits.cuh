// float64 products on the bf16 tensor cores by exact digits.
//
// A vector of float64 values with largest biased exponent e is held as 61-bit integers
// f = round(v 2^(1083 - e)), |f| < 2^61 (values within eight binades of the largest are exact), and
// these as seven balanced digits of nine bits, f = sum_s q_s 2^(9 (6 - s)), |q_s| <= 256, which bf16
// holds exactly.  Digit products are integers below 2^16, so a float32 accumulator adds them exactly
// while their sum stays below 2^24; products with s + t = d share an accumulator, and d = 0 .. 6 are
// kept (what is dropped is below 2^-58 of the product of the two largest magnitudes, per term,
// against float64's own rounding of 2^-53).  The seven accumulators v_d of an entry are combined in
// integers, T = sum_d v_d 2^(9 (6 - d)), and rounded once to float64: no float64 arithmetic, which on
// GB300 takes 16 cycles per warp instruction.
//
// A vector that holds an infinity or a NaN is marked by exponent 2047; its results are NaN.
#pragma once

#include <stdint.h>

#include "sep_plane.cuh"

namespace dig {

constexpr int ND = 7;                             // digits

__device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// the seven digits of v against the largest exponent e of its vector, as the high halves of float32
// bit patterns (bf16), digit s in q[s]
__device__ __forceinline__ void split(double v, int e, uint32_t (&q)[ND]) {
    const long long b = __double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7ff), down = e - ev - 8;
    long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    if (down <= 0) m <<= -down;
    else m = down < 62 ? ((m >> (down - 1)) + 1) >> 1 : 0;
    if (ev == 0) m = 0;                           // zeros and subnormals
    if (b < 0) m = -m;
#pragma unroll
    for (int s = ND - 1; s >= 0; --s) {
        const int lo = s > 0 ? (((int)m + 256) & 511) - 256 : (int)m;
        m = (m - lo) >> 9;
        q[s] = __float_as_uint(__int_as_float(0x4b400000 + lo) - 12582912.f) >> 16;
    }
}

// (hi 2^27 + lo) 2^e rounded to float64 (to nearest, ties away from zero; subnormal results are zero)
__device__ __forceinline__ double combine(long long hi, long long lo, int e) {
    long long H = hi + (lo >> 27);
    uint32_t rem = (uint32_t)lo & 0x7ffffffu;
    const bool neg = H < 0;
    if (neg) {
        H = -H - (rem ? 1 : 0);
        rem = (0x8000000u - rem) & 0x7ffffffu;
    }
    if (H == 0) {
        if (rem == 0) return 0.0;
        H = rem;
        rem = 0;
        e -= 27;
    }
    const int lz = __clzll(H);
    const unsigned long long M =
        ((unsigned long long)H << lz) | (lz >= 27 ? (unsigned long long)rem << (lz - 27) : (unsigned long long)rem >> (27 - lz));
    const unsigned long long mant = (M >> 11) + ((M >> 10) & 1);
    const int ex = 38 - lz + e + 52 + 1023;
    unsigned long long bits = ((unsigned long long)ex << 52) + (mant - 0x10000000000000ull);
    if (ex <= 0) bits = 0;
    if (ex >= 2046) bits = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

}  // namespace dig
