// Device helpers for kernels that walk the cube's entries (readback, zeroing,
// continuum subtraction): conversions and float-pair arithmetic that stay off the
// FP64 pipe (about two lanes a clock and SM on GB300: widening, adding and
// narrowing the four sums of every entry of a 6.7e7-entry cube took 1.3 ms there,
// three times its memory time), and 32-byte accesses.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace vista {

// Four doubles of one cube entry (32-byte aligned) in one access.
struct Double4 {
    double x, y, z, w;
};
__device__ __forceinline__ Double4 load_double4(const double *p)
{
    Double4 d;
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(d.x), "=d"(d.y), "=d"(d.z), "=d"(d.w) : "l"(p));
    return d;
}
__device__ __forceinline__ void store_zero32(void *p)
{
    asm volatile("st.global.v4.b64 [%0], {%1, %1, %1, %1};" ::"l"(p), "l"(0ll) : "memory");
}

// The mixed cube's master entries are zero but for those that a checkpoint or a
// fold has moved sums into (about one touched entry in eight after a stack of six
// reductions an entry); a bit per entry says which may not be, so that the other
// masters' 32 bytes are neither read nor zeroed.
__device__ __forceinline__ bool is_moved(uint32_t word, int64_t i) { return (word >> (i & 31)) & 1u; }

// A double as hi + lo, two floats: hi is the double truncated to 24
// significant bits, lo the remaining 29 bits rounded to a float (so hi + lo
// is the double to about 2^-47 relative, less where lo falls below the
// normal floats).  Integer and FP32 operations only.  Magnitudes below 2^-126
// give (0, 0): zero, and values far below any sum of weights or visibilities.
// Magnitudes from 2^128 on, infinities and NaNs give a pair that is not finite
// (the exponent saturates; with a branch for them the subtraction of an FP64 cube
// of 1.7e7 entries took 290 us instead of 263).
__device__ __forceinline__ float2 split_double(double d)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e < 897) return make_float2(0.f, 0.f);
    const unsigned sign = (unsigned)(b >> 63) << 31, ef = (unsigned)min(e - 896, 255) << 23;
    const unsigned hi_bits = sign | ef | ((unsigned)(b >> 29) & 0x7fffffu);
    // the low 29 mantissa bits times 2^-52 (exact), times 2^(e - 1023)
    const float lo = (__uint2float_rn((unsigned)(b & 0x1fffffffu)) * 0x1p-52f) * __uint_as_float(ef);
    return make_float2(__uint_as_float(hi_bits), sign ? -lo : lo);
}

__device__ __forceinline__ float2 add_ff(float2 a, float b)   // (a.x + a.y) + b as a pair
{
    const float t = a.x + b, z = t - a.x;
    const float err = (a.x - (t - z)) + (b - z);
    const float lo = a.y + err, hi = t + lo;
    return make_float2(hi, lo - (hi - t));
}

// A float as a double and a double rounded to a float (to nearest, ties to even),
// by moving the fields: integer instructions, where the FP64 unit's conversions
// are as slow as its additions.
static __device__ __noinline__ double widen_slow(float x) { return (double)x; }    // subnormal, infinite, NaN
static __device__ __noinline__ float narrow_slow(double x) { return (float)x; }    // outside the normal floats
__device__ __forceinline__ double widen_exact(float x)
{
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (__builtin_expect(e - 1u >= 254u && (b << 1) != 0u, 0)) return widen_slow(x);
    return __hiloint2double((int)((b & 0x80000000u) | (e ? ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3) : 0u)), (int)(b << 29));
}
__device__ __forceinline__ float narrow(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
    if (__builtin_expect((uint32_t)(m >> 52) - 897u > 253u, 0)) return narrow_slow(x);
    const uint32_t f = (uint32_t)((m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29) - (896u << 23);   // (may round up to infinity)
    return __uint_as_float(f | ((uint32_t)(b >> 32) & 0x80000000u));
}

// An entry's FP32 partials c and FP64 master sums m, added in FP64 and rounded
// to floats.  Four FP64 operations: only entries with a master pay them (one
// touched entry in eight as a rule), beside the memory's time.
__device__ __forceinline__ float4 sum_f32(float4 c, const Double4 &m)
{
    return make_float4(narrow(widen_exact(c.x) + m.x), narrow(widen_exact(c.y) + m.y), narrow(widen_exact(c.z) + m.z),
                       narrow(widen_exact(c.w) + m.w));
}

}  // namespace vista
