// dg_intfp64.cuh -- IEEE binary64 multiplication, division and square root, round to
// nearest even, on the integer ALU.
//
// This GPU issues an FP64 instruction from a warp once every 64 cycles per SM
// sub-partition (0.5e12 lane operations/s over the chip, measured), while its integer
// ALU retires more than a warp instruction every other cycle.  An FP64 multiply costs
// about 28 integer instructions here, a division or a square root about 60
// (the compiler's FP64 division and square root are each a sequence of FP64
// instructions), so kernels bound by the FP64 pipe run these operations on the integer
// ALU, beside the additions that stay on the FP64 pipe.  Measured on a line contraction
// s += D F of length 6 (multiply and add rounded separately): 0.25e12 pairs/s with both
// on the FP64 pipe, 0.50e12 with the multiplies here, which is the rate of the FP64
// additions alone.
//
// Results are the correctly rounded ones, the same bits as the FP64 unit's.  The fast
// paths cover normal operands with normal results; everything else (zeros, subnormals,
// infinities, NaN, results outside the normal range) takes the FP64 instruction.
//
// Methods, from the definitions: the multiply forms the exact 128-bit product of the
// two significands.  The division is long division in two digits with a reciprocal
// estimate from below, an exact remainder after every digit, and one final correction;
// a quotient of two 53-bit significands is never half-way between two 53-bit values,
// so floor(2^53 q) decides the rounding.  The square root refines an estimate from
// the exact remainder v - s^2 and corrects the last bit against it; a root is never
// half-way either.
#pragma once

#include <cstdint>
#include <cstring>
#include <cmath>
#if !defined(__CUDACC__)
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace dg {
namespace ifp {

// The bits of a double.  (Assembly on the device: given a plain cast the compiler turns
// tests of these bits back into FP64 comparisons.)
__host__ __device__ __forceinline__ uint64_t dbits(double x)
{
#ifdef __CUDA_ARCH__
    uint32_t h, l;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "d"(x));
    return ((uint64_t)h << 32) | l;
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

__host__ __device__ __forceinline__ double bdbl(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}

__host__ __device__ __forceinline__ uint32_t hi32(uint64_t b) { return (uint32_t)(b >> 32); }
__host__ __device__ __forceinline__ uint32_t lo32(uint64_t b) { return (uint32_t)b; }
__host__ __device__ __forceinline__ uint64_t mk64(uint32_t h, uint32_t l) { return ((uint64_t)h << 32) | l; }
__host__ __device__ __forceinline__ uint64_t mulw(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// 1/x and 1/sqrt(x) in FP32.  What the digits below are exact for: 1/x within 2^-22 absolute for x
// in [1, 2] (divisor() takes that much off, to stay below), 1/sqrt(x) within 2^-22.5 relative
// (root_fast's second remainder then stays within 2^53).  The PTX manual gives the instructions'
// largest errors as 2^-23 on that range, and 2^-22.9 relative.
__host__ __device__ __forceinline__ float rcp_est(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

__host__ __device__ __forceinline__ float rsqrt_est(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / std::sqrt(x);
#endif
}

__host__ __device__ __forceinline__ uint32_t fbits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    std::memcpy(&b, &x, 4);
    return b;
#endif
}

__host__ __device__ __forceinline__ float bflt(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    std::memcpy(&x, &b, 4);
    return x;
#endif
}

// The FP64 instructions of the rare paths, as calls: inlined, the compiler executes
// them every time and selects, and an FP64 instruction holds its pipe even with every
// lane predicated off.
#ifdef __CUDACC__
static __device__ __noinline__ double slow_mul(double a, double b) { return __dmul_rn(a, b); }
static __device__ __noinline__ double slow_div(double a, double b) { return __ddiv_rn(a, b); }
static __device__ __noinline__ double slow_root(double x) { return __dsqrt_rn(x); }
#endif
#ifdef __CUDA_ARCH__
#define DG_IFP_SLOW(device_expr, host_expr) device_expr
#else
#define DG_IFP_SLOW(device_expr, host_expr) host_expr
#endif

// ---------------------------------------------------------------------------
// A factor prepared for products: the 53-bit significand shifted left by 11 (top bit
// set; zero for a zero) in h:l, and in e the high word's sign and exponent fields.
struct Factor {
    uint32_t h, l, e;
};

__host__ __device__ __forceinline__ Factor factor(double x)
{
    const uint64_t b = dbits(x);
    const uint32_t H = hi32(b), L = lo32(b);
    Factor f;
    f.h = (H << 11) | (L >> 21) | 0x80000000u;
    f.l = L << 11;
    f.e = H & 0xfff00000u;
    if ((H & 0x7ff00000u) == 0u) f.h = f.l = 0u;  // zero (subnormals are excluded by factor_ok)
    return f;
}

// Whether a factor is in the range the products below are exact for: zero, or an
// exponent field within 500 of the bias (no product of two such factors over- or
// underflows).
__host__ __device__ __forceinline__ bool factor_ok(double x)
{
    const uint64_t b = dbits(x);
    const uint32_t m = hi32(b) << 1;  // exponent and significand, no sign
    return (m - (523u << 21) < (1001u << 21)) | ((m | lo32(b)) == 0u);
}

// RN(f d) for two factors that factor_ok accepts, a zero product as +0.
__host__ __device__ __forceinline__ double mul_unsigned_zero(const Factor &f, const Factor &d)
{
    const uint64_t p0 = mulw(f.l, d.l);
    const uint64_t p1 = mulw(f.h, d.l) + hi32(p0);
    const uint64_t p2 = mulw(f.l, d.h) + lo32(p1);
    uint64_t T = mulw(f.h, d.h) + hi32(p1) + hi32(p2);  // top 64 bits of the product
    const uint32_t th = hi32(T);
    const uint32_t n = th >> 31;  // 1: the product of the significands is >= 2
    // the bits of the lower 64 folded into the lowest one (below the rounding position)
    const uint32_t rest = lo32(p2) | lo32(p0);
    T |= rest != 0u ? 1u : 0u;
    // to nearest even at bit 10 + n: half an ulp less one, plus the bit kept last (the
    // top 64 bits of a product end at least 2^12 below 2^64, so nothing carries out)
    T += (0x1ffu + (n << 9)) + ((uint32_t)(T >> (10 + n)) & 1u);
    // sign and exponent fields of the product, the exponent less 1 (the significand's
    // leading bit adds it back; a rounding carry into 2^53 raises it by itself)
    const uint32_t e = f.e + (d.e - (1024u << 20)) + (n << 20);
    return bdbl((T >> (10 + n)) + mk64(th == 0u ? 0u : e, 0u));
}

// RN(f d), the sign of a zero product included.
__host__ __device__ __forceinline__ double mul(const Factor &f, const Factor &d)
{
    const uint64_t b = dbits(mul_unsigned_zero(f, d));
    return bdbl(b | mk64((f.e ^ d.e) & 0x80000000u, 0u));
}

// RN(a b).  (The fast result is formed first and replaced where an operand is out of
// range: the factors of an operand used several times are then prepared once.)
__host__ __device__ __forceinline__ double mul(double a, double b)
{
    double r = mul(factor(a), factor(b));
    if (!(factor_ok(a) & factor_ok(b))) r = DG_IFP_SLOW(slow_mul(a, b), a * b);
    return r;
}

// ---------------------------------------------------------------------------
// RN(a / b): significands A, B in [2^52, 2^53); A doubled if below B, so that the
// quotient is in [1, 2).  r = 2^84 / B from below, within 2^-30 relative.  Digits of 28
// and 25 bits: q = floor-ish(rem 2^k / B), never above the true digit and below it by
// less than 2 (rem's truncation costs 1/4, r 1/2, the floor 1), rem exact (modulo 2^64,
// always below 2^54).  Several quotients by one divisor share its part.
struct Divisor {
    double b;
    uint64_t B;
    uint32_t nl, nh;  // -B
    uint32_t r;
    uint32_t h;       // high word of b
};

__host__ __device__ __forceinline__ Divisor divisor(double b)
{
    Divisor d;
    const uint64_t bb = dbits(b);
    d.b = b;
    d.h = hi32(bb);
    const uint32_t Bh = (d.h & 0xfffffu) | 0x100000u, Bl = lo32(bb);
    d.B = mk64(Bh, Bl);
    // reciprocal of B's significand rounded up to FP32, y in [0.5, 1], as 2^32 y less
    // 2^10 (2^-22 of it, no less than the estimate's error): r0 <= 2^84 / B
    const uint32_t c = (Bh << 11) | (Bl >> 21);  // B 2^-21, in [2^31, 2^32)
    const float y = rcp_est(bflt((c >> 8) + 0x3f000001u));
    const uint32_t r0 = (fbits(y) << 8) + 0x7ffffc00u;
    // one Newton step: r0 (1 + e) with e = 1 - (c + 1) r0 2^-63 in (0, 2^-19), no more
    // than the true error
    const uint64_t e = 0x8000000000000000ULL - (mulw(c, r0) + r0);
    d.r = r0 + (hi32(mulw((uint32_t)(e >> 12), r0)) >> 19);
    d.nl = 0u - Bl;
    d.nh = ~Bh + (Bl == 0u ? 1u : 0u);
    return d;
}

// RN(a / b) where div_ok (a in the middle of the exponent range or zero, b in the
// middle of it: normal operands, normal quotient).
__host__ __device__ __forceinline__ bool div_ok(double a, const Divisor &d)
{
    const uint64_t ab = dbits(a);
    const uint32_t m = hi32(ab) << 1;
    return ((m - (523u << 21) < (1001u << 21)) | ((m | lo32(ab)) == 0u)) & ((d.h << 1) - (523u << 21) < (1001u << 21));
}

__host__ __device__ __forceinline__ double div_fast(double a, const Divisor &d)
{
    const uint64_t ab = dbits(a);
    const uint32_t ah = hi32(ab);
    uint64_t rem = mk64((ah & 0xfffffu) | 0x100000u, lo32(ab));
    // exponent field of the quotient less 1
    uint32_t ex = (ah & 0x7ff00000u) - (d.h & 0x7ff00000u) + (1022u << 20);
    if (rem < d.B) {
        rem <<= 1;
        ex -= 1u << 20;
    }
    const uint32_t q1 = hi32(mulw((uint32_t)(rem >> 22), d.r)) >> 2;
    rem <<= 28;
    rem += mulw(q1, d.nl) + mk64(q1 * d.nh, 0u);
    const uint32_t q2 = hi32(mulw((uint32_t)(rem >> 22), d.r)) >> 5;
    rem <<= 25;
    rem += mulw(q2, d.nl) + mk64(q2 * d.nh, 0u);
    uint64_t Q = ((uint64_t)q1 << 25) + q2;  // floor(2^53 A/B), or one below
    Q += rem >= d.B ? 2u : 1u;                                      // corrected, plus the rounding 1
    uint64_t bits = mk64(ex, 0u) + (Q >> 1);
    if ((ah & 0x7ff00000u) == 0u) bits = 0u;  // a = 0
    return bdbl(bits | mk64((ah ^ d.h) & 0x80000000u, 0u));
}

__host__ __device__ __forceinline__ double div(double a, const Divisor &d)
{
    double r = div_fast(a, d);
    if (!div_ok(a, d)) r = DG_IFP_SLOW(slow_div(a, d.b), a / d.b);
    return r;
}

__host__ __device__ __forceinline__ double div(double a, double b) { return div(a, divisor(b)); }

// ---------------------------------------------------------------------------
// RN(sqrt(x)): v = x scaled by an even power of two into [1, 4), V = 2^52 v.  With
// y ~ 1/sqrt(v) (FP32): S1 = 2^24 sqrt(v) from y, the exact remainder V - S1^2 2^4
// gives the next bits through y/2, twice; then floor(2^53 sqrt v) is fixed against the
// exact remainder.
__host__ __device__ __forceinline__ bool root_ok(double x) { return (hi32(dbits(x)) >> 20) - 1u <= 2045u; }  // positive, normal

__host__ __device__ __forceinline__ double root_fast(double x)
{
    const uint64_t xb = dbits(x);
    const uint32_t xh = hi32(xb);
    const uint32_t ef = xh >> 20, odd = (ef & 1u) ^ 1u;  // odd power of two: v in [2, 4)
    const uint64_t V = mk64((xh & 0xfffffu) | 0x100000u, lo32(xb)) << odd;  // 2^52 v
    // FP32 copy of v (truncated) and 1/sqrt
    const float vf = bflt(((127u + odd) << 23) + ((xh & 0xfffffu) << 3) + (lo32(xb) >> 29));
    const float y = rsqrt_est(vf);                  // in (0.5, 1]
    const float s = vf * y;                          // sqrt(v), in [1, 2), to 2^-21
    const uint32_t yi = (uint32_t)(int32_t)(y * 1073741824.0f);  // 2^30 y
    const uint32_t S1 = (uint32_t)(int32_t)(s * 16777216.0f);    // 2^24 sqrt(v) + d, |d| < 16
    // remainder R1 = 2^48 v - S1^2, times 2^4 (V = 2^52 v): |R1 2^4| < 2^34
    const int64_t R1 = (int64_t)V - (int64_t)(mulw(S1, S1) << 4);
    // next 22 bits: R1 2^22 / (2 S1) = (R1 2^4) 2^18 / 2^25 / (S1 2^-24) = (R1 2^4) y 2^-7
    const int32_t t1 = (int32_t)(R1 >> 3);                       // |t1| < 2^31
    const int32_t d1 = (int32_t)(((int64_t)t1 * (int64_t)yi) >> 34);
    const uint64_t S2 = ((uint64_t)S1 << 22) + (int64_t)d1;      // 2^46 sqrt(v), within 2^5
    // remainder R2 = 2^92 v - S2^2 = V 2^40 - S2^2 (modulo 2^64; |R2| < 2^53)
    const uint32_t s2h = hi32(S2), s2l = lo32(S2);
    const uint64_t sq = mulw(s2l, s2l) + mk64(2u * s2h * s2l, 0u);  // S2^2 modulo 2^64
    const int64_t R2 = (int64_t)((V << 40) - sq);
    // next 7 bits: R2 2^7 / (2 S2) = R2 2^6 2^-46 y = (R2 2^-22) (2^30 y) 2^-48
    const int32_t t2 = (int32_t)(R2 >> 22);
    const int32_t d2 = (int32_t)(((int64_t)t2 * (int64_t)yi) >> 48);
    uint64_t F = (S2 << 7) + (int64_t)d2;                        // 2^53 sqrt(v), within 1
    // exact: 2^106 v - F^2 = V 2^54 - F^2 modulo 2^64 (|.| < 2^57)
    const uint32_t fh = hi32(F), fl = lo32(F);
    int64_t R = (int64_t)((V << 54) - (mulw(fl, fl) + mk64(2u * fh * fl, 0u)));
    F += R < 0 ? 0u : (R > (int64_t)(2u * F) ? 2u : 1u);  // floor + 1 (the rounding)
    const uint32_t ex = (ef - odd + 1023u) >> 1;
    return bdbl(mk64((ex - 1u) << 20, 0u) + (F >> 1));
}

__host__ __device__ __forceinline__ double root(double x)
{
    double r = root_fast(x);
    if (!root_ok(x)) r = DG_IFP_SLOW(slow_root(x), std::sqrt(x));
    return r;
}

// ---------------------------------------------------------------------------
// RN(a + b) / 2 of two operands without sign, where half_sum_ok: the larger one normal
// and neither it nor the sum near the ends of the range, the smaller one normal or zero.
__host__ __device__ __forceinline__ bool half_sum_ok(double a, double b)
{
    const uint64_t x = dbits(a), y = dbits(b), big = x > y ? x : y, small = x > y ? y : x;
    return ((hi32(big) >> 20) - 2u <= 2042u) & (((hi32(small) >> 20) - 1u <= 2043u) | (small == 0u));
}

__host__ __device__ __forceinline__ double half_sum_fast(double a, double b)
{
    const uint64_t x = dbits(a), y = dbits(b), big = x > y ? x : y, small = x > y ? y : x;
    const uint32_t ex = hi32(big) >> 20, d = ex - (hi32(small) >> 20), sh = d < 63u ? d : 63u;
    // significands with their top bits at bit 62, the smaller one aligned, the bits it
    // loses folded into the lowest one
    const uint64_t A = ((big & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    const uint64_t B = small == 0u ? 0u : ((small & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    uint64_t T = A + (B >> sh);
    T |= ((B >> sh) << sh) != B ? 1u : 0u;
    const uint32_t n = (uint32_t)(T >> 63);
    T += (0x1ffu + (n << 9)) + ((uint32_t)(T >> (10 + n)) & 1u);  // to nearest even at bit 10 + n
    return bdbl((T >> (10 + n)) + mk64((ex + n - 2u) << 20, 0u));
}

// Whether |a - b| <= 2^-48 a (difference and bound rounded), where close_ok: b without
// sign and finite, a positive, normal and so is the bound, and the two in one binade
// (bit patterns then count their distance in ulps; the bound is 16 to 31 ulps) or more
// than 64 patterns apart (more than the bound, also where a binade's end halves the ulp).
__host__ __device__ __forceinline__ bool close_ok(double a, double b)
{
    const uint64_t x = dbits(a), y = dbits(b);
    const bool in = ((hi32(x) >> 20) - 49u <= 1997u) & ((hi32(y) >> 20) <= 2046u);
    return in & (((hi32(x) ^ hi32(y)) >> 20 == 0u) | (x - y + 64u > 128u));
}

__host__ __device__ __forceinline__ bool close_fast(double a, double b)
{
    const uint64_t x = dbits(a), y = dbits(b);
    const uint32_t t = 16u + ((hi32(x) >> 16) & 15u);
    return x - y + t <= 2u * t;
}

// ---------------------------------------------------------------------------
// fmin / fmax by comparing the bit patterns (negatives ordered in reverse), for
// operands that are not NaN.
__host__ __device__ __forceinline__ int64_t order_key(double x)
{
    const int64_t b = (int64_t)dbits(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

__host__ __device__ __forceinline__ bool finite(double x) { return (hi32(dbits(x)) & 0x7fffffffu) < 0x7ff00000u; }

// ---------------------------------------------------------------------------
// The arithmetic a formula is written for.  Fast runs these operations on the integer
// ALU and notes in `ok` whether every operand was in range; a formula evaluated with it
// is evaluated again with Native, in a call, where it was not.  One check per formula
// keeps the FP64 instructions of the rare case behind one branch.  (Products that are
// zero come out as +0.)
struct Fast {
    using Div = Divisor;
    bool ok = true;
    __host__ __device__ __forceinline__ double mul(double a, double b)
    {
        ok = ok & factor_ok(a) & factor_ok(b);
        return mul_unsigned_zero(factor(a), factor(b));
    }
    __host__ __device__ __forceinline__ Div divisor(double b) { return ifp::divisor(b); }
    __host__ __device__ __forceinline__ double div(double a, const Div &d)
    {
        ok = ok & div_ok(a, d);
        return div_fast(a, d);
    }
    __host__ __device__ __forceinline__ double div(double a, double b) { return div(a, divisor(b)); }
    __host__ __device__ __forceinline__ double root(double x)
    {
        ok = ok & root_ok(x);
        return root_fast(x);
    }
    __host__ __device__ __forceinline__ double least(double a, double b)
    {
        ok = ok & finite(a) & finite(b);
        return order_key(a) < order_key(b) ? a : b;
    }
    __host__ __device__ __forceinline__ double greatest(double a, double b)
    {
        ok = ok & finite(a) & finite(b);
        return order_key(a) > order_key(b) ? a : b;
    }
    __host__ __device__ __forceinline__ bool positive(double x)
    {
        ok = ok & finite(x);
        return (int64_t)dbits(x) > 0;
    }
};

#ifdef __CUDACC__
struct Native {
    using Div = double;
    __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    __device__ __forceinline__ double divisor(double b) { return b; }
    __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    __device__ __forceinline__ double root(double x) { return __dsqrt_rn(x); }
    __device__ __forceinline__ double least(double a, double b) { return fmin(a, b); }
    __device__ __forceinline__ double greatest(double a, double b) { return fmax(a, b); }
    __device__ __forceinline__ bool positive(double x) { return x > 0.0; }
};
#endif

}  // namespace ifp
}  // namespace dg
