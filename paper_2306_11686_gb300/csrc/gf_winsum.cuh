/*
 * Sums of doubles on the integer pipe, exact while the values' exponents lie
 * in a window of 32 binades.
 *
 * A compensated FP64 addition takes five FP64 operations, and GB300 retires
 * about 1.7 of them per clock and SM: a sum over 2^26 doubles took 680 us,
 * eight times what reading them takes (101 to 109 us like this).  Here a value whose biased exponent e
 * has p = e - base in [0, 31] is the 53-bit significand shifted left by p,
 * added (its one's complement for a negative value, whose missing +1s are
 * counted) to a 96-bit integer in units of 2^(base - 1075): about 16 integer
 * instructions, no rounding.  With 53 + 31 bits a term, 2^11 terms fit: the
 * one that opens a window and GF_WIN_TERMS more, after which the accumulator
 * is folded into a double pair.  (Fixed-point accumulation in
 * the manner of U. Kulisch, "Computer Arithmetic and Validity", with a short
 * register that moves.)
 *
 * Values outside the window (zeros aside) go to the caller's compensated FP64
 * sum.  The window moves to them where that pays: emptying the integer takes
 * up to 18 FP64 operations, and the other lanes of the warp wait for them, so
 * values that are spread over more binades than the window holds must not move
 * it to and fro (2^26 values spread over 40 to 600 binades took 4.5 to 4.7 ms
 * when every larger value and every eighth smaller one did, 0.56 to 0.60 now, and
 * 0.68 ms with the compensated sum alone).  It moves
 *  - up, for a larger value among the first two misses, while it holds few
 *    terms (the first value was a small one);
 *  - to the sixteenth miss in a row, with no term between them, where all of
 *    these lie in one window (the data have drifted).
 * Windows end below 2^909: sums near overflow, infinities and NaNs keep the
 * FP64 sum's behaviour.
 *
 * Host and device, so the CPU tests compare it with exact sums.
 */
#ifndef GF_WINSUM_CUH
#define GF_WINSUM_CUH
#include "gf_intpipe.cuh"

#define GF_WIN_TERMS 2047u       /* terms between two folds, besides one that add_out adds */
#define GF_WIN_TOP 1900u         /* highest exponent that makes a window */

struct gf_winsum {
    uint32_t w0, w1, w2, neg;    /* the sum's words; negative terms */
    uint32_t base;               /* window (0: none yet) */
    uint32_t run, cand, seen;    /* misses in a row that lie in window cand; the room at the last one */
    uint32_t early;              /* misses left that may move the window up at once */

    GF_IP_HD gf_winsum() : w0(0), w1(0), w2(0), neg(0), base(0), run(0), cand(0), seen(0), early(2) {}

    static GF_IP_HD uint32_t base_of(uint32_t e) { return (e - 15u) & ~15u; }

    /* the first window, for values of which e is the highest exponent */
    GF_IP_HD void open(uint32_t e)
    {
        if (e >= 32u && e <= GF_WIN_TOP)
            base = base_of(e);
    }

    /* p of x: 0 .. 31 inside the window */
    GF_IP_HD uint32_t place(double x) const
    {
        return ((uint32_t)(gf_ip_bits(x) >> 52) & 0x7ffu) - base;
    }

    /* x with place(x) = p <= 31 and base >= 1 */
    GF_IP_HD void add_in(double x, uint32_t p)
    {
        const uint64_t b = gf_ip_bits(x);
        const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, mh = (hi & 0xfffffu) | 0x100000u;
        const uint32_t s = (uint32_t)((int32_t)hi >> 31);
#ifdef __CUDA_ARCH__
        const uint32_t t0 = (lo << p) ^ s, t1 = __funnelshift_l(lo, mh, p) ^ s, t2 = __funnelshift_l(mh, 0u, p) ^ s;
        asm("add.cc.u32 %0, %0, %3; addc.cc.u32 %1, %1, %4; addc.u32 %2, %2, %5;"
            : "+r"(w0), "+r"(w1), "+r"(w2)
            : "r"(t0), "r"(t1), "r"(t2));
#else
        const uint64_t m = (uint64_t)mh << 32 | lo;
        const uint32_t t0 = (lo << p) ^ s, t1 = (uint32_t)((m << p) >> 32) ^ s, t2 = (p ? mh >> (32u - p) : 0u) ^ s;
        uint64_t c = (uint64_t)w0 + t0;
        w0 = (uint32_t)c;
        c = (uint64_t)w1 + t1 + (c >> 32);
        w1 = (uint32_t)c;
        w2 += t2 + (uint32_t)(c >> 32);
#endif
        neg -= s;
    }

    /* the integer as 96-bit two's complement */
    GF_IP_HD void words(uint32_t *v) const
    {
        uint64_t c = (uint64_t)w0 + neg;
        v[0] = (uint32_t)c;
        c = (uint64_t)w1 + (c >> 32);
        v[1] = (uint32_t)c;
        v[2] = w2 + (uint32_t)(c >> 32);
    }

    /* a 128-bit two's complement integer in units of 2^(base - 1075), as up to four exact doubles.  A low
     * window's scale is subnormal, and its products are exact all the same. */
    template <class ADD> static GF_IP_HD void pieces(const uint32_t *v, uint32_t base, ADD add)
    {
        const uint32_t s = (uint32_t)((int32_t)v[3] >> 31);
        uint32_t m[4];
        uint64_t c = s & 1u;
        for (int k = 0; k < 4; k++) {
            c += v[k] ^ s;
            m[k] = (uint32_t)c;
            c >>= 32;
        }
        for (int k = 3; k >= 0; k--) {
            if (m[k] == 0u)
                continue;
            double x = (double)m[k];
            int e = (int)base - 1075 + 32 * k;
            if (e < -1022) {                     /* in two steps */
                x *= gf_ip_double((uint64_t)(1023 - 512) << 52);
                e += 512;
            }
            x *= gf_ip_double((uint64_t)(e + 1023) << 52);
            add(s ? -x : x);
        }
    }

    /* empty the integer: ADD(double) gets its pieces */
    template <class ADD> GF_IP_HD void fold(ADD add)
    {
        uint32_t v[4];
        words(v);
        v[3] = (uint32_t)((int32_t)v[2] >> 31);
        w0 = w1 = w2 = neg = 0;
        if (base)
            pieces(v, base, add);
    }

    /* a value that place() puts outside the window (or the first one).  room: what is left of GF_WIN_TERMS, which
     * tells whether a term came in since the last miss.  Bases are multiples of 16, so that threads whose values
     * are alike share theirs and their integers can be added. */
    template <class ADD> GF_IP_HD void add_out(double x, ADD add, uint32_t room = 0)
    {
        const uint64_t b = gf_ip_bits(x);
        if ((b & 0x7fffffffffffffffull) == 0)
            return;
        const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;
        if (e < 32u || e > GF_WIN_TOP) {
            add(x);
            return;
        }
        if (base) {
            if (run == 0u || room != seen || e - cand > 31u) {
                run = 0u;
                cand = base_of(e);
            }
            run++;
            seen = room;
            const bool up = early != 0u && e > base && GF_WIN_TERMS - room < 8u;
            early -= early != 0u ? 1u : 0u;
            if (!up && run < 16u) {
                add(x);
                return;
            }
            fold(add);
            base = cand;
            run = 0u;
        } else {
            base = base_of(e);
        }
        add_in(x, e - base);
    }
};

#endif
