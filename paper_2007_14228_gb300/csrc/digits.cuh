// float64 products on the bf16 tensor cores by integer digits.
//
// A vector of float64 values with largest biased exponent e is held as 61-bit integers
// f = round(v 2^(1083 - e)), |f| < 2^61 (values within eight binades of the largest are exact), and
// these as seven balanced digits of nine bits, f = sum_s q_s 2^(9 (6 - s)), |q_s| <= 256, which bf16
// holds exactly.  Digit products are integers below 2^16, so a float32 accumulator adds them exactly
// while their sum stays below 2^24; products with s + t = d share an accumulator, and d = 0 .. 6 are
// kept.  The seven accumulators v_d of an entry are combined in integers, T = sum_d v_d 2^(9 (6 - d)),
// and rounded once to float64: no float64 arithmetic, which on GB300 takes 16 cycles per warp
// instruction.
//
// Error: a term loses six digit products of up to 2^16 at weight 2^45 and less below, and up to half a
// unit of either f times the other, together below 7.01 2^61 where the product of the two largest
// magnitudes is 2^120 at least.  The accumulator d = 6 passes 2^24 from 43 terms on, and a unit lost there
// weighs 2^54.  A sum of p <= 48 terms is therefore off by at most
//   7.2 p 2^-59 x (power of two of the first vector's largest) x (that of the second's).
// For entries far smaller than that, which a float64 sum would hold to 2^-53 of their own
// terms, the callers compare it with sum |a||b| and add in float64 where it is too coarse: `magnitude`
// gives the bf16 factors of one more product that bounds the sum of magnitudes from below.
//
// A vector that holds an infinity or a NaN has exponent 2047, one of subnormal values only counts as 1,
// and 0 means that all are zero; the callers do not use the digits where values or results could be
// subnormal or infinite.
#pragma once

#include <stdint.h>

#include "sep_plane.cuh"

namespace dig {

constexpr int ND = 7;                             // digits

__device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ bool nonzero(double v) { return (__double_as_longlong(v) << 1) != 0; }

// |v| 2^(1023 - e) cut to eight bits, as bf16 bits: zero below 2^-126 (e >= 128), at most 2^60
__device__ __forceinline__ uint32_t magnitude(double v, int e) {
    return (uint32_t)min(max(((__double2hiint(v) & 0x7fffffff) >> 13) - ((e - 127) << 7), 0), 187 << 7);
}

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

// (hi 2^SH + lo) 2^e rounded to float64 (to nearest, ties away from zero; subnormal results, which the
// callers do not ask for, are zero)
template <int SH>
__device__ __forceinline__ double combine(long long hi, long long lo, int e) {
    constexpr uint32_t LOW = SH == 32 ? 0xffffffffu : (1u << (SH & 31)) - 1u;
    long long H = hi + (lo >> SH);
    uint32_t rem = (uint32_t)lo & LOW;
    const bool neg = H < 0;
    if (neg) {
        H = -H - (rem ? 1 : 0);
        rem = (0u - rem) & LOW;
    }
    if (H == 0) {
        if (rem == 0) return 0.0;
        H = rem;
        rem = 0;
        e -= SH;
    }
    const int lz = __clzll(H);
    const unsigned long long M =
        ((unsigned long long)H << lz) | (lz >= SH ? (unsigned long long)rem << (lz - SH) : (unsigned long long)rem >> (SH - lz));
    const unsigned long long mant = (M >> 11) + ((M >> 10) & 1);
    const int ex = 63 - lz + SH + e + 1023;
    unsigned long long bits = ((unsigned long long)ex << 52) + (mant - 0x10000000000000ull);
    if (ex <= 0) bits = 0;
    if (ex >= 2047) bits = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

// Eight digits of eight bits, for sums over many rows (digit products are below 2^14, so 64 of them
// in each of eight pairs stay exact; pairs with s + t > 7 are dropped, below 2^-57 of the product of the
// two largest magnitudes per term): f = round(v 2^(1084 - e)), |f| < 2^62, f = sum_s q_s 2^(8 (7 - s)),
// -128 <= q_s < 128.  With 128 added to every digit they are the bytes of one integer.  Byte s of the
// result (from the top) is q_s + 128.
constexpr int NB = 8;

__device__ __forceinline__ unsigned long long bytes_of(double v, int e) {
    const long long b = __double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7ff), down = e - ev - 9;
    long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    if (down <= 0) m <<= -down;
    else m = down < 62 ? ((m >> (down - 1)) + 1) >> 1 : 0;
    if (ev == 0) m = 0;                           // zeros and subnormals
    if (b < 0) m = -m;
    return (unsigned long long)m + 0x8080808080808080ull;
}

// byte k of w, less 128, as the bits of a float32 (its high half is the bf16)
__device__ __forceinline__ uint32_t digit_of(uint32_t w, int k) {
    return __float_as_uint(__uint_as_float(__byte_perm(w, 0x4b000000u, 0x7650u | (uint32_t)k)) - 8388736.f);
}

}  // namespace dig
