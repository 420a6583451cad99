// Quotients rounded to codes: two at a time, without the general division.
//
// fl(x / s) for a divisor with few significant bits (an fp16 scale has 11, a 6-bit multiple of one 17) in three operations,
// given inv = fl(1 / s): a product and one correction step (P. Markstein,
// Computation of elementary functions on the IBM RISC System/6000, 1990).  p = fl(x * inv) is off by 2^-23 relative at most; the remainder x - p*s is exact in one fma (it is
// a multiple of 2^-39 of x, and at most 2^-22 of it); p + remainder * inv, before its rounding, is off by 2^-46 relative
// at most.  That rounds like x / s itself: the middle m between two neighbouring fp32 values has 25 significant bits, so
// m*s is never x (24 bits), x - m*s is a multiple of 2^-41 of x, and x / s is no closer to m than that.  Valid for finite x
// and s, no overflow or underflow on the way (weights and scales are fp16 values or their small multiples).
#pragma once

namespace spqt {

__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\tfma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// Divisors of two groups; 0 divides everything to 0.
struct Divisor2 {
    float2 minus, inv;

    __device__ __forceinline__ Divisor2() {}
    __device__ __forceinline__ explicit Divisor2(float2 s)
    {
        minus = make_float2(-s.x, -s.y);
        inv = make_float2(s.x != 0.0f ? __frcp_rn(s.x) : 0.0f, s.y != 0.0f ? __frcp_rn(s.y) : 0.0f);
    }
    __device__ __forceinline__ float2 quotient(float2 x) const
    {
        const float2 p = mul2(x, inv);
        return fma2(fma2(p, minus, x), inv, p);
    }
};

// v in [0, 2^22) rounded to the nearest integer, ties to even: the integers are the low bits of the words
__device__ __forceinline__ float2 round_to_low_bits(float2 v) { return add2(v, make_float2(12582912.0f, 12582912.0f)); }

// the low bytes of four words
__device__ __forceinline__ unsigned four_bytes(float a, float b, float c, float d)
{
    return __byte_perm(__byte_perm(__float_as_uint(a), __float_as_uint(b), 0x0040), __byte_perm(__float_as_uint(c), __float_as_uint(d), 0x0040), 0x5410);
}

}  // namespace spqt
