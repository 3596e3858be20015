/*
 * Sums of a few non-negative doubles, each add correctly rounded as the FP64
 * add rounds it, computed on the FP32 pipe.
 *
 * GB300 retires about 1.7 FP64 adds per clock and SM and 128 FP32
 * instructions.  An FP64 add emulated here takes eight instructions, seven of
 * them FP32, so a stencil whose FP64 adds bound it runs several times faster
 * on exact FP32 arithmetic.  The scheme:
 *
 *  - a value x whose binary exponent lies in a window of nine binades
 *    [top - 8, top] (or x = +0) is an integer X < 2^61 in units of
 *    2^(top - 60).  It is cut into three chunks, each a float that holds an
 *    integer multiple of its lattice:
 *        a: X bits 60..40 (lattice 2^40), b: bits 39..19 (2^19), c: bits 18..0 (1),
 *    so the chunks of up to six values add without rounding (6 * 2^21 < 2^24);
 *  - the exponent e of a sum a + b + c is the exponent of
 *    d = RZ(a + RZ(b + c)): every chunk is non-negative, truncation to a
 *    lattice that divides a's lattice cannot step over a power of two, so d
 *    and the exact sum lie in the same binade;
 *  - the sum's ulp is 2^(e - 52) units (1 to 2^11: below b's lattice), and
 *    rounding the sum to it is rounding c: with M = 2^(e - 29),
 *    c' = RN(c + M) - M is c rounded to a multiple of ulp(M) = 2^(e - 52),
 *    ties to even, since c < 2^22 <= M.  M is d's exponent field scaled by
 *    2^-29, folded into the two multiply-adds.  a and b are even multiples
 *    of that ulp, so ties fall as they do for the whole sum;
 *  - a value outside the window makes chunk a a NaN, which every sum it
 *    enters carries to the end, where one test sends the point to the
 *    ordinary FP64 path.
 *
 * gf_fix_div6 rounds the sum / 6 to a double: with the significand n scaled
 * so that n / 3 has 53 bits, n / 3 is never half way between two integers, so
 * the rounded quotient is floor((n + 1) / 3), a multiplication by the
 * reciprocal (T. Granlund, P. Montgomery, "Division by invariant integers
 * using multiplication", PLDI 1994).
 *
 * Host and device, so the CPU tests compare it with IEEE arithmetic.
 */
#ifndef GF_FIXSUM_CUH
#define GF_FIXSUM_CUH
#include "gf_intpipe.cuh"
#ifndef __CUDA_ARCH__
#include <cfenv>
#include <cmath>
#endif

GF_IP_HD float gf_fs_float(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}
GF_IP_HD uint32_t gf_fs_word(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    memcpy(&b, &x, 4);
    return b;
#endif
}
GF_IP_HD float gf_fs_fma(float x, float y, float z)
{
#ifdef __CUDA_ARCH__
    return __fmaf_rn(x, y, z);
#else
    return fmaf(x, y, z);
#endif
}
GF_IP_HD float gf_fs_add_rz(float x, float y)
{
#ifdef __CUDA_ARCH__
    return __fadd_rz(x, y);
#else
    const int m = fegetround();
    fesetround(FE_TOWARDZERO);
    volatile float p = x, q = y;
    volatile float r = p + q;
    fesetround(m);
    return r;
#endif
}
/* (hi:lo << k) >> 32, k clamped to 32 */
GF_IP_HD uint32_t gf_fs_shl(uint32_t lo, uint32_t hi, uint32_t k)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_lc(lo, hi, k);
#else
    return k >= 32u ? lo : (uint32_t)(((((uint64_t)hi << 32) | lo) << k) >> 32);
#endif
}
/* x << k, 0 from k = 32 on */
GF_IP_HD uint32_t gf_fs_shl1(uint32_t x, uint32_t k)
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(k));
    return r;
#else
    return k >= 32u ? 0u : x << k;
#endif
}
/* low word of hi:lo >> k, 0 <= k <= 31 */
GF_IP_HD uint32_t gf_fs_shr(uint32_t lo, uint32_t hi, uint32_t k)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(lo, hi, k);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> k);
#endif
}
/* leading zeros of x; 2^32 - 1 for x = 0 */
GF_IP_HD uint32_t gf_fs_clz(uint32_t x)
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
#else
    return x ? (uint32_t)__builtin_clz(x) : 0xffffffffu;
#endif
}

/* floor((hi:lo) / 3) for hi < 2^30: four 32 x 32 -> 64 multiply-adds */
GF_IP_HD uint64_t gf_fs_third(uint32_t lo, uint32_t hi)
{
    const uint64_t w0 = (uint64_t)lo * 0x55555556u;
    const uint64_t w1 = (uint64_t)lo * 0x55555555u + (uint32_t)(w0 >> 32);
    const uint64_t w2 = (uint64_t)hi * 0x55555556u + w1;
    return (uint64_t)hi * 0x55555555u + (uint32_t)(w2 >> 32);
}

/* The highest window's top: its values lie below 2^(2044 - 1023) = 2^1021, so six of them sum below 2^1024.  One
 * binade higher the FP64 sum can overflow to infinity, and the chunks' sum does not. */
#define GF_FIX_TOP 2043u

struct gf_fix3 {
    float a, b, c;
};

/* x in chunks; elow = the biased exponent of the window's lowest binade */
GF_IP_HD gf_fix3 gf_fix_split(double x, uint32_t elow)
{
    const uint64_t bits = gf_ip_bits(x);
    const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
    const uint32_t k = (hi >> 20) - elow;             /* 0 .. 8 inside the window (a sign bit is outside) */
    const float base = k > 8u && (hi | lo) != 0u ? gf_fs_float(0x7fffffffu) : -9223372036854775808.0f;   /* -2^63 */
    const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
    /* X = m << k, below 2^61; +0 has k beyond 32 and the clamped shifts leave 0 */
    const uint32_t xh = gf_fs_shl(lo, mh, k), xl = gf_fs_shl1(lo, k);
    gf_fix3 r;
    /* 2^23 + integer by its bits, then scaled and the 2^23 taken off */
#ifdef __CUDA_ARCH__
    const uint32_t ab = __byte_perm(xh, 0x4bu, 0x4321);
#else
    const uint32_t ab = 0x4b000000u | (xh >> 8);
#endif
    r.a = gf_fs_fma(gf_fs_float(ab), 1099511627776.0f, base);                                        /* 2^40 */
    r.b = gf_fs_fma(gf_fs_float(0x4b000000u | (gf_fs_shr(xl, xh, 19u) & 0x1fffffu)), 524288.0f, -4398046511104.0f);
    r.c = gf_fs_float(0x4b000000u | (xl & 0x7ffffu)) - 8388608.0f;
    return r;
}

/* x + y, rounded to 53 bits (ties to even) */
GF_IP_HD gf_fix3 gf_fix_add(gf_fix3 x, gf_fix3 y)
{
    gf_fix3 r;
    r.a = x.a + y.a;
    r.b = x.b + y.b;
    const float c = x.c + y.c;
    const float d = gf_fs_add_rz(r.a, gf_fs_add_rz(r.b, c));
    const float m = gf_fs_float(gf_fs_word(d) & 0x7f800000u);
    r.c = gf_fs_fma(m, -1.862645149230957e-09f, gf_fs_fma(m, 1.862645149230957e-09f, c));          /* 2^-29 */
    return r;
}

/* the sum is a number of the window's units, not NaN (0 where all its values are +0) */
GF_IP_HD bool gf_fix_ok(gf_fix3 t) { return t.a >= 0.0f; }

/* RN(t / 6) for a sum t of at most six values with gf_fix_ok, each add rounded */
GF_IP_HD double gf_fix_div6(gf_fix3 t, uint32_t elow)
{
    /* T in units, 0 or 2^52 <= T < 6 * 2^61 < 2^64 */
    const uint64_t bc = (uint64_t)(uint32_t)(t.b * 1.9073486328125e-06f) * 524288u + (uint32_t)t.c;
    const uint32_t th = (uint32_t)(bc >> 32) + (uint32_t)(t.a * 2.3283064365386963e-10f), tl = (uint32_t)bc;
    /* at most 11; T = 0 takes the z that makes the result's exponent field 0 (elow >= 5), and all shifts leave 0 */
    const uint32_t zt = gf_fs_clz(th), z = zt < elow + 7u ? zt : elow + 7u;
    const uint32_t nh = gf_fs_shl(tl, th, z), nl = gf_fs_shl1(tl, z);          /* leading bit at 63, 11 zero bits below */
    const uint32_t s = nh < 0xc0000000u ? 9u : 10u;                  /* n = T 2^z >> s: n / 3 in [2^52, 2^53) */
    const uint32_t qh = nh >> s, ql = gf_fs_shr(nl, nh, s);
    /* nearest integer to n / 3 = floor((n + 1) / 3): the high half of (n + 1) (2^64 + 2) / 3, exact below
     * 2^63; n is even, so n + 1 is n | 1 */
    const uint64_t n = gf_fs_third(ql | 1u, qh);
    /* biased exponent elow + 10 - z - k, with k = 11 - s; n carries the hidden bit */
    return gf_ip_double(n + ((uint64_t)(elow + s - z - 2u) << 52));
}

#endif
