// Fixed-point arithmetic of the refined weight solve: 64-bit integers on the
// integer pipe for the quantities that must be known beyond double precision
// (kernel values r^3, monomials, residuals).  On this GPU the FP64 units issue
// 2 lanes per clock per SM and the integer multiply-add pipe 64, so a 64-bit
// fixed-point product (three 32 x 32 -> 64 multiplies) takes a fraction of
// the time of a DMUL and carries more bits: the coordinates lie in the unit
// disk, so every quantity has a known bound and needs no exponent.
//
//   coordinate  X = x 2^61            |x| <= 1
//   r^2         q = r^2 2^58          r <= 2
//   r           s = r 2^60
//   r^3         v = value 2^56        r^3 <= 8
//   p_k         v = value 2^61        |p_k| <= 1
//
// A 64-bit value is split into two signed 32-bit digits v = hi 2^32 + lo, so
// that every partial product is a signed 32 x 32 -> 64 multiply-add.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rbffd {

struct Digits {
    int hi, lo;
};

__host__ __device__ __forceinline__ Digits fx_digits(int64_t v) {
    Digits d;
    d.lo = (int)(uint32_t)(uint64_t)v;
    d.hi = (int)(uint32_t)((uint64_t)v >> 32) + (int)((uint32_t)d.lo >> 31);  // lo signed: carry its sign into hi
    return d;
}

__host__ __device__ __forceinline__ int64_t fx_mul32(int a, int b) { return (int64_t)a * b; }

// Bit casts and shifts that mean the same on host and device.
__host__ __device__ __forceinline__ float fx_as_float(uint32_t b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    union { uint32_t u; float f; } c;
    c.u = b;
    return c.f;
#endif
}
__host__ __device__ __forceinline__ uint32_t fx_as_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    union { uint32_t u; float f; } c;
    c.f = f;
    return c.u;
#endif
}
// f 2^k, k in [-126, 127], exact for normal results
__host__ __device__ __forceinline__ float fx_pow2f(int k) { return fx_as_float((uint32_t)(k + 127) << 23); }

// Nearest integer of f, |f| < 2^22, and back (|v| < 2^22): the sum with
// 1.5 2^23 has the integer in its low fraction bits.  (The conversion
// instructions run at a quarter of the rate.)
__host__ __device__ __forceinline__ int fx_small_int(float f) {
    return (int)(fx_as_bits(f + 12582912.0f) - 0x4B400000u);
}
__host__ __device__ __forceinline__ float fx_small_float(int v) {
    return fx_as_float((uint32_t)v + 0x4B400000u) - 12582912.0f;
}

// Nearest integer, saturating at the int32 range.
__host__ __device__ __forceinline__ int fx_round(float f) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(f);
#else
    return f >= 2147483520.0f ? 0x7fffffff : (f <= -2147483520.0f ? -0x7fffffff : (int)__builtin_rintf(f));
#endif
}

// x 2^61 of a double |x| < 4 (bits below 2^-61 truncated), by integer
// instructions; 0 where |x| < 2^-62.
__host__ __device__ __forceinline__ int64_t fx_coord(uint64_t bits) {
    const int e = (int)((bits >> 52) & 0x7ff);
    const uint64_t m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    const int sh = e - (1023 - 61 + 52);  // value = m 2^(e - 1023 - 52)
    uint64_t v = sh >= 0 ? m << (sh & 63) : (sh > -54 ? m >> ((-sh) & 63) : 0ull);
    return (bits >> 63) ? -(int64_t)v : (int64_t)v;
}

// r^2 2^58 of the coordinate differences (each |.| <= 2^62): the leading
// digits' squares plus the cross terms; the lowest partial products
// (< 2^-58 in all) are dropped.
__host__ __device__ __forceinline__ int64_t fx_r2(int64_t dx, int64_t dy) {
    const Digits x = fx_digits(dx), y = fx_digits(dy);
    const int64_t a = fx_mul32(x.hi, x.hi) + fx_mul32(y.hi, y.hi);   // unit 2^-58
    const int64_t c = fx_mul32(x.hi, x.lo) + fx_mul32(y.hi, y.lo);   // unit 2^-90, counted twice
    return a + (c >> 31);
}

// r 2^60 from q = r^2 2^58, its float value qf and yf ~ 1/r (relative errors
// <= ~2^-16).  Three digits: s0 = qf yf to 2^-21, then twice the Newton
// correction (r^2 - s^2) yf / 2 of the exact integer remainder, to 2^-42 and
// 2^-60.  Below r ~ 2^-8 the last digits lose accuracy as 2^-50 / r; r^3
// (whose error is r^2 times that of r) stays exact to its unit.
__host__ __device__ __forceinline__ int64_t fx_sqrt(int64_t q, float qf, float yf) {
    const float hy = 0.5f * yf;
    const int s0 = fx_small_int(qf * yf * 0x1p21f);                       // unit 2^-21
    const int64_t e0 = q - (int64_t)((uint64_t)fx_mul32(s0, s0) << 16);   // r^2 - s0^2, unit 2^-58
    const float d1f = (float)(int)(e0 >> 12) * 0x1p-46f * hy;
    const int d1 = fx_small_int(d1f * 0x1p42f);                           // unit 2^-42
    const int64_t e1 = e0 - (fx_mul32(s0, d1) >> 4) - (fx_mul32(d1, d1) >> 26);
    const float d2f = fx_small_float((int)e1) * 0x1p-58f * hy;
    const int d2 = fx_round(d2f * 0x1p60f);
    return (int64_t)(((uint64_t)(int64_t)s0 << 39) + ((uint64_t)(int64_t)d1 << 18)) + d2;
}

// r^3 2^56 of q = r^2 2^58 and s = r 2^60.
__host__ __device__ __forceinline__ int64_t fx_cube(int64_t q, int64_t s) {
    const Digits a = fx_digits(q), b = fx_digits(s);
    const int64_t h = fx_mul32(a.hi, b.hi);                               // unit 2^-54
    const int64_t c = fx_mul32(a.hi, b.lo) + fx_mul32(a.lo, b.hi);        // unit 2^-86
    return (int64_t)((uint64_t)h << 2) + (c >> 30);
}

// x p 2^61 of a coordinate and a monomial (2^61 both), |x p| <= 1.
__host__ __device__ __forceinline__ int64_t fx_mono(const Digits& x, const Digits& p) {
    const int64_t h = fx_mul32(x.hi, p.hi);                               // unit 2^-58
    const int64_t c = fx_mul32(x.hi, p.lo) + fx_mul32(x.lo, p.hi);        // unit 2^-90
    return (int64_t)((uint64_t)h << 3) + (c >> 29);
}

}  // namespace rbffd
