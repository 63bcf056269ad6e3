// Integer-built conversions between floating point and fixed-point digits
// (internal header): used wherever a matrix is cut into 8-bit digit slices
// for the tensor cores or an exact integer sum is turned back into FP64.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace gb {

// Library fallback of the integer-built conversions below, for results
// outside the normal double range.  Kept out of line: inlined, the compiler
// may evaluate it on every element (its int -> double conversion and scaling
// run on the FP64 pipe) and select the result afterwards.
static __device__ __noinline__ double ldexp_i64_slow(long long t, int e) { return ldexp(static_cast<double>(t), e); }

// T * 2^e rounded to the nearest double (ties to even), i.e. the value of
// ldexp((double)T, e), for |T| < 2^63, built with integer operations (the
// FP64 pipe retires two operations per clock and SM); results outside the
// normal exponent range take the library path.
__device__ __forceinline__ double scaled_i64_to_f64(long long T, int e)
{
    if (T == 0) return 0.0;
    const unsigned long long sign = T < 0 ? (1ull << 63) : 0ull;
    const unsigned long long u = T < 0 ? 0ull - static_cast<unsigned long long>(T) : static_cast<unsigned long long>(T);
    const int lz = __clzll(static_cast<long long>(u));
    int msb = 63 - lz;
    const unsigned long long m = u << lz;  // leading one at bit 63
    unsigned long long keep = m >> 11;     // 53 significant bits
    const unsigned long long rem = m & 0x7FFull;
    if (rem > 0x400ull || (rem == 0x400ull && (keep & 1ull))) keep++;
    if (keep >> 53) {  // rounded up to the next power of two
        keep >>= 1;
        msb++;
    }
    const int ex = msb + e;
    if (ex < -1022 || ex > 1023) return ldexp_i64_slow(T, e);
    return __longlong_as_double(static_cast<long long>(sign | (static_cast<unsigned long long>(ex + 1023) << 52) |
                                                       (keep & ((1ull << 52) - 1))));
}

// Biased binary exponent field of a double (0 for zero / subnormal).
__device__ __forceinline__ int bexp(double a)
{
    return int((static_cast<unsigned long long>(__double_as_longlong(a)) >> 52) & 0x7FF);
}

// Balanced base-256 digit of x: the d in [-128, 127] with d = x (mod 256).
__device__ __forceinline__ int bal8(int x) { return ((x + 128) & 255) - 128; }
// The FP32 bit pattern of an integer |d| < 2^22, exactly: d added to the
// integer bits of 1.5 2^23 adds d to that value, which is then subtracted.
__device__ __forceinline__ uint32_t small_int_f32bits(int d)
{
    return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f);
}
// Two BF16 in one word from FP32 patterns whose low 16 bits are zero (the
// high halves are then the BF16 values exactly): lo_elem first.
__device__ __forceinline__ uint32_t pack_hi16(uint32_t lo_elem, uint32_t hi_elem)
{
    return __byte_perm(lo_elem, hi_elem, 0x7632);
}

}  // namespace gb
