/* Host check of gf_winsum.cuh at its limit: the value that opens a window,
 * then more terms than fit between two folds, all at the window's top with
 * full significands.  Every place that the opening value can take, both signs
 * and a window that opens again on the way; the total is compared with the
 * exact integer.
 *
 *   winsum_limit_check          prints "sums checked N mismatches M" */
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include "gf_winsum.cuh"

int main()
{
    long long n = 0, bad = 0;
    for (int p = 15; p <= 30; p++)
        for (int terms : {2046, 2047, 2048, 2049, 5000})
            for (double sign : {1.0, -1.0})
                for (int late : {0, 1}) {
                    gf_winsum w;
                    uint32_t room = GF_WIN_TERMS;
                    /* all values are multiples of 2^-20 below 2^33: the sums below are exact integers */
                    __int128 want = 0, got = 0;
                    auto out = [&](double y) { got += (__int128)ldexp(y, 60); };
                    auto put = [&](double x) {
                        want += (__int128)ldexp(x, 60);
                        const uint32_t at = w.place(x);
                        if (at <= 31u && w.base) {          /* as a thread's part of a reduction adds */
                            w.add_in(x, at);
                            if (--room == 0u) {
                                w.fold(out);
                                room = GF_WIN_TERMS;
                            }
                        } else {
                            w.add_out(x, out);
                        }
                    };
                    if (late)                               /* a window far below, left for the next value's */
                        for (int k = 0; k < 3; k++)
                            put(sign * 0x1p-40);
                    put(sign * ldexp(2.0 - 0x1p-52, p - 15));          /* exponent 1023 + p - 15: place p */
                    const double top = ldexp(2.0 - 0x1p-52, 16);       /* the highest exponent of that window */
                    for (int k = 0; k < terms; k++)
                        put(sign * top);
                    w.fold(out);
                    n++;
                    bad += want != got;
                }
    printf("sums checked %lld mismatches %lld\n", n, bad);
    return bad != 0;
}
