// Conversions and signs of FP64 values by integer instructions.  On this GPU an
// FP64 conversion holds the FP64 pipe as long as a multiply-add (16 clocks a warp),
// which bounds the kernels that use these.
#pragma once

namespace tl {

__device__ __forceinline__ double flip(double v, bool sign)  // sign ? -v : v, no FP64 instruction
{
    return __hiloint2double(__double2hiint(v) ^ (sign ? (int)0x80000000u : 0), __double2loint(v));
}

__device__ __forceinline__ double widen_bits(float v)  // (double)v
{
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    const int s = __clz((int)m) - 8;  // subnormal: the shift that brings its first bit to bit 23
    const bool small = m < 0x800000u;
    const unsigned f = small ? m << (s & 31) : m;
    const unsigned e = small ? (unsigned)(896 - s) << 20 : m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
    const unsigned hi = m ? (small ? e + (f >> 3) : (f >> 3) + e) : 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(f << 29));
}

__device__ __forceinline__ float narrow_bits(double v)  // (float)v: to nearest, ties to even
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)(hi >> 20 & 0x7ffu) - 896;  // the FP32 exponent field
    const unsigned long long m = ((unsigned long long)(hi & 0xfffffu | 0x100000u) << 32) | lo;
    const int shift = e >= 1 ? 29 : e > -30 ? 30 - e : 60;  // subnormal: more bits go
    const unsigned long long r = m >> shift, rest = m & ((1ull << shift) - 1), half = 1ull << (shift - 1);
    unsigned f = (unsigned)r + (rest > half || (rest == half && (r & 1)) ? 1u : 0u);
    if (e >= 1) f += (unsigned)(e - 1) << 23;  // f has the leading bit: a carry reaches the exponent
    if (e >= 255) f = e == 2047 - 896 && (m & 0xfffffffffffffull) ? 0x7fffffffu : 0x7f800000u;
    return __uint_as_float(f | (hi & 0x80000000u));
}

}  // namespace tl
