// IEEE binary64 multiplication, division, square root and conversions with round-to-nearest-even,
// evaluated with integer instructions only.  A value is held as
// (-1)^neg m 2^e with m = 0 (zero) or 2^52 <= m < 2^53, so every result is
// the one the FP64 unit returns for the same operands (IEEE 754 binary64,
// roundTiesToEven) for finite operands whose results stay normal; the
// callers keep to that range and fall back to FP64 instructions outside it.
// On this GPU FP64 instructions, conversions included, issue at 1/64 of the
// FP32 rate, so the FP64 collision kernel takes this path for the rounding of its
// weights, its divisions and its square roots.
// The header also compiles as plain C++ (the host unit test checks it
// against the host's double arithmetic).
#pragma once
#include <cstdint>
#include <cstring>
#include <cmath>

#ifndef __CUDACC__
#define BZ_HD inline
#else
#define BZ_HD __host__ __device__ __forceinline__
#endif

namespace bz {

struct Exact64 {
    uint64_t m;  // 0, or 2^52 <= m < 2^53
    int e;       // value = m 2^e
    int neg;
};

BZ_HD int clz64(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

BZ_HD uint64_t umulhi64(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// Rounds m 2^-sh (1 <= sh <= 63) to the nearest integer, ties to even.
BZ_HD uint64_t shr_rne(uint64_t m, int sh)
{
    const uint64_t q = m >> sh;
    const uint64_t rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    return q + ((rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull);
}

// (double)n, rounded to nearest even when |n| >= 2^53.
BZ_HD Exact64 x64_from_ll(long long n)
{
    Exact64 r;
    r.neg = n < 0;
    const uint64_t a = r.neg ? 0ull - (uint64_t)n : (uint64_t)n;
    if (a == 0) {
        r.m = 0;
        r.e = 0;
        return r;
    }
    const int nb = 64 - clz64(a);  // bit length
    if (nb <= 53) {
        r.m = a << (53 - nb);
        r.e = nb - 53;
    } else {
        int sh = nb - 53;
        uint64_t m = shr_rne(a, sh);
        if (m == (1ull << 53)) {
            m >>= 1;
            ++sh;
        }
        r.m = m;
        r.e = sh;
    }
    return r;
}

// The exact value of a finite double.
BZ_HD Exact64 x64_from_double(double d)
{
    uint64_t b;
    memcpy(&b, &d, sizeof b);
    Exact64 r;
    r.neg = (int)(b >> 63);
    const int be = (int)((b >> 52) & 0x7ffu);
    const uint64_t frac = b & ((1ull << 52) - 1ull);
    if (be == 0) {  // zero (subnormals do not occur in the callers' range)
        r.m = 0;
        r.e = 0;
    } else {
        r.m = frac | (1ull << 52);
        r.e = be - 1075;
    }
    return r;
}

BZ_HD double x64_to_double(Exact64 x)
{
    uint64_t b = (uint64_t)x.neg << 63;
    if (x.m) b |= ((uint64_t)(x.e + 1075) << 52) | (x.m & ((1ull << 52) - 1ull));
    double d;
    memcpy(&d, &b, sizeof d);
    return d;
}

// a * b rounded to nearest even (a zero operand gives a signed zero).
BZ_HD Exact64 x64_mul(Exact64 a, Exact64 b)
{
    Exact64 r;
    r.neg = a.neg ^ b.neg;
    if (a.m == 0 || b.m == 0) {
        r.m = 0;
        r.e = 0;
        return r;
    }
    // the 105- or 106-bit product hi 2^64 + lo, cut to 53 bits
    const uint64_t hi = umulhi64(a.m, b.m), lo = a.m * b.m;
    int sh = (hi >> 41) ? 53 : 52;
    uint64_t m = (hi << (64 - sh)) | (lo >> sh);
    const uint64_t rem = lo & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    m += (rem > half || (rem == half && (m & 1ull))) ? 1ull : 0ull;
    if (m == (1ull << 53)) {
        m >>= 1;
        ++sh;
    }
    r.m = m;
    r.e = a.e + b.e + sh;
    return r;
}

// u x rounded to nearest even, for an integer 0 < u < 2^53 (exactly a
// double) and a nonzero x: the product of the two doubles.
BZ_HD Exact64 x64_mul_u(uint64_t u, Exact64 x)
{
    Exact64 r;
    r.neg = x.neg;
    const uint64_t hi = umulhi64(u, x.m), lo = u * x.m;
    const int nb = hi ? 128 - clz64(hi) : 64 - clz64(lo);  // bit length of the product (>= 53)
    const int sh = nb - 53;                                // 0 .. 53
    uint64_t m;
    if (sh == 0) {
        m = lo;
    } else {
        m = (hi << (64 - sh)) | (lo >> sh);
        const uint64_t rem = lo & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
        m += (rem > half || (rem == half && (m & 1ull))) ? 1ull : 0ull;
    }
    int e = x.e + sh;
    if (m == (1ull << 53)) {
        m >>= 1;
        ++e;
    }
    r.m = m;
    r.e = e;
    return r;
}

// llrint(x 2^k), rounded to nearest even; false when |x 2^k| >= 2^62 (the
// caller then uses the FP64 conversion).
BZ_HD bool x64_rint_scaled(Exact64 x, int k, long long* out)
{
    if (x.m == 0) {
        *out = 0;
        return true;
    }
    const int s = x.e + k;
    uint64_t v;
    if (s >= 0) {
        if (s > 9) return false;  // m 2^s >= 2^62
        v = x.m << s;
    } else if (s >= -63) {
        v = shr_rne(x.m, -s);
    } else {
        v = 0;  // below 2^-10: rounds to 0
    }
    *out = x.neg ? -(long long)v : (long long)v;
    return true;
}

// Quotient and square root of binary64 values, correctly rounded, by integer digits
// (20, 20 and 13 bits) whose estimates come from one FP32 reciprocal (root): the
// remainders are exact in 64-bit arithmetic, so an estimate that is off by one only
// makes the next remainder larger, and the last remainder's sign gives the floor of the
// 54-bit result.  Rounding it is adding 1 and dropping the last bit: neither a
// quotient nor a root of 53-bit numbers lies halfway between two of them.
// Error of a digit in its units: quotient 1.32, 0.99 and 0.51, root 0.91, 1.9 and 0.51
// with estimates good to 2^-21.9 (two units in the last place and the operand's
// truncation); the remainders fit with room.
#ifndef X64_RCP
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float x64_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float x64_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
#define X64_RCP(x) x64_rcp(x)
#define X64_RSQRT(x) x64_rsqrt(x)
#else
#define X64_RCP(x) (1.0f / (x))
#define X64_RSQRT(x) (1.0f / sqrtf(x))
#endif
#endif

BZ_HD float x64_float(uint32_t bits)
{
    float f;
    memcpy(&f, &bits, sizeof f);
    return f;
}
// nearest integer of x y for |x y| < 2^22
BZ_HD int x64_digit(float x, float y)
{
    const float t = fmaf(x, y, 12582912.0f);  // 1.5 2^23
    uint32_t b;
    memcpy(&b, &t, sizeof b);
    return (int)(b - 0x4B400000u);
}

// a / b; false (out unset) unless both and the quotient are safely normal
BZ_HD bool x64_div(uint64_t a, uint64_t b, uint64_t& out)
{
    const uint64_t frac = (1ull << 52) - 1ull;
    const uint32_t ea = (uint32_t)(a >> 52) & 0x7FFu, eb = (uint32_t)(b >> 52) & 0x7FFu;
    const int e = (int)ea - (int)eb + 1023;
    if (ea - 1u >= 2046u || eb - 1u >= 2046u || (unsigned)(e - 2) >= 2044u) return false;
    const uint64_t ma = (a & frac) | (1ull << 52), mb = (b & frac) | (1ull << 52);
    const bool lt = ma < mb;  // quotient of the mantissas below 1: doubled
    const float y = X64_RCP(x64_float(0x3F800000u | ((uint32_t)(b >> 29) & 0x7FFFFFu)));
    const int q1 = x64_digit(x64_float(0x3F800000u | ((uint32_t)(a >> 29) & 0x7FFFFFu)), y * (lt ? 2097152.0f : 1048576.0f));
    const uint64_t r1 = (ma << (lt ? 21 : 20)) - (uint64_t)((long long)q1 * (long long)mb);
    const int q2 = x64_digit((float)(int)((long long)r1 >> 23), y * 0.001953125f);  // 2^(23 - 52 + 20)
    const uint64_t r2 = (r1 << 20) - (uint64_t)((long long)q2 * (long long)mb);
    const int q3 = x64_digit((float)(int)((long long)r2 >> 23), y * 1.52587890625e-5f);  // 2^(23 - 52 + 13)
    const uint64_t r3 = (r2 << 13) - (uint64_t)((long long)q3 * (long long)mb);
    const uint64_t Q = ((uint64_t)(long long)q1 << 33) + ((uint64_t)(long long)q2 << 13) + (uint64_t)(long long)(q3 - (int)(r3 >> 63));
    out = ((a ^ b) & (1ull << 63)) + ((uint64_t)(uint32_t)(e - 1 - (int)lt) << 52) + ((Q + 1) >> 1);
    return true;
}

// sqrt(a); false (out unset) unless a is +-0 or normal and positive
BZ_HD bool x64_sqrt(uint64_t a, uint64_t& out)
{
    if ((a << 1) == 0) {
        out = a;
        return true;
    }
    const uint32_t ea = (uint32_t)(a >> 52);  // with the sign: 2048 and more if negative
    if (ea - 1u >= 2046u) return false;
    const uint32_t odd = (ea + 1u) & 1u;  // parity of the exponent ea - 1023
    const uint64_t A = ((a & ((1ull << 52) - 1ull)) | (1ull << 52)) << odd;
    const float af = x64_float((0x3F800000u + (odd << 23)) | ((uint32_t)(a >> 29) & 0x7FFFFFu));
    const float y = X64_RSQRT(af);
    const int s1 = x64_digit(af, y * 1048576.0f);
    const long long r1 = (long long)(A - ((uint64_t)((long long)s1 * s1) << 12));
    const int d2 = x64_digit((float)(int)(r1 >> 4), y * 0.001953125f);  // 2^(4 - 13)
    const long long r2 = (long long)(((uint64_t)r1 << 28) - ((uint64_t)((long long)s1 * d2) << 21) - (uint64_t)((long long)d2 * d2));
    const int d3 = x64_digit((float)(int)(r2 >> 13), y * 3.0517578125e-5f);  // 2^(13 - 28)
    const long long S2 = ((long long)s1 << 20) + d2;
    const uint64_t r3 = ((uint64_t)r2 << 26) - ((uint64_t)(S2 * d3) << 14) - (uint64_t)((long long)d3 * d3);
    const uint64_t Q = ((uint64_t)S2 << 13) + (uint64_t)(long long)(d3 - (int)(r3 >> 63));
    out = ((uint64_t)(((ea + 1023u - odd) >> 1) - 1u) << 52) + ((Q + 1) >> 1);
    return true;
}

// a b; false (out unset) unless one is +-0 and the other finite, or both and the product
// are safely normal
BZ_HD bool x64_mul(uint64_t a, uint64_t b, uint64_t& out)
{
    const uint32_t ah = (uint32_t)(a >> 32), bh = (uint32_t)(b >> 32), a0 = (uint32_t)a, b0 = (uint32_t)b;
    const uint32_t ea = (ah >> 20) & 0x7FFu, eb = (bh >> 20) & 0x7FFu, sign = (ah ^ bh) & 0x80000000u;
    const int e = (int)(ea + eb) - 1023;  // of a product of mantissas in [1, 2)
    if (ea - 1u >= 2046u || eb - 1u >= 2046u || (unsigned)(e - 2) >= 2043u) {
        const bool az = (a << 1) == 0, bz = (b << 1) == 0;
        if (!((az && eb != 0x7FFu) || (bz && ea != 0x7FFu))) return false;
        out = (uint64_t)sign << 32;
        return true;
    }
    const uint32_t a1 = (ah & 0xFFFFFu) | 0x100000u, b1 = (bh & 0xFFFFFu) | 0x100000u;
    const uint64_t p0 = (uint64_t)a0 * b0;
    uint64_t mid = (uint64_t)a1 * b0 + (p0 >> 32);
    mid = (uint64_t)a0 * b1 + mid;
    uint64_t top = (uint64_t)a1 * b1 + (mid >> 32);  // product = top 2^64 + (mid mod 2^32) 2^32 + (p0 mod 2^32)
    const uint32_t lo = (uint32_t)p0, ml = (uint32_t)mid;
    const int two = (int)((uint32_t)(top >> 41) & 1u);  // mantissa product >= 2
    const int sh = 20 + two;                            // bits of ml below the result
    const uint64_t m = (top << (32 - sh)) | (ml >> sh);
    const uint32_t half = 1u << (sh - 1), rest = ml & (2u * half - 1u);
    const bool up = rest > half || (rest == half && (lo != 0u || (m & 1u)));
    out = ((uint64_t)(sign + ((uint32_t)(e - 1 + two) << 20)) << 32) + m + (up ? 1u : 0u);
    return true;
}

#ifdef __CUDACC__
static __device__ __noinline__ double mul64_slow(double a, double b) { return a * b; }
static __device__ __noinline__ double mul64(double a, double b)
{
    uint64_t o;
    if (x64_mul((uint64_t)__double_as_longlong(a), (uint64_t)__double_as_longlong(b), o)) return __longlong_as_double((long long)o);
    return mul64_slow(a, b);
}
static __device__ __noinline__ double div64_slow(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt64_slow(double a) { return sqrt(a); }
// a / b and sqrt(a) as the FP64 instructions give them, without those: some 70 integer
// and FP32 instructions (150 cycles) for nine or ten of 64 cycles.  Calls, not inlined: a
// root's dozen copies overflow the instruction cache (7 species, 12 x 13 x 10: 1.07 against
// 0.88 ms).
static __device__ __noinline__ double div64(double a, double b)
{
    uint64_t o;
    if (x64_div((uint64_t)__double_as_longlong(a), (uint64_t)__double_as_longlong(b), o)) return __longlong_as_double((long long)o);
    return div64_slow(a, b);
}
static __device__ __noinline__ double sqrt64(double a)
{
    uint64_t o;
    if (x64_sqrt((uint64_t)__double_as_longlong(a), o)) return __longlong_as_double((long long)o);
    return sqrt64_slow(a);
}
#endif

}  // namespace bz
