/* Host check of gf_fixsum.cuh at the highest windows: sums of six values of
 * the window's upper binades, each add rounded as IEEE rounds it (also to
 * infinity), and their sixths.
 *
 *   fixsum_top_check TOP   prints "div6 checked N mismatches M, highest window H" */
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "gf_fixsum.cuh"

int main(int argc, char **argv)
{
    const uint32_t top = argc > 1 ? (uint32_t)atoi(argv[1]) : 0u, elow = top - 8u;
    uint64_t rng = 11;
    auto rnd = [&] {
        uint64_t z = (rng += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    long long n = 0, bad = 0;
    for (int it = 0; it < 200000; it++) {
        double x[6];
        for (int k = 0; k < 6; k++) {
            const uint64_t m = it % 3 == 0 ? 0xfffffffffffffull - (rnd() & 3) : rnd() & 0xfffffffffffffull;
            const uint64_t b = (uint64_t)(top - (it % 2 ? rnd() % 3 : 0)) << 52 | m;
            memcpy(&x[k], &b, 8);
        }
        gf_fix3 t = gf_fix_split(x[0], elow);
        volatile double v = x[0];
        for (int k = 1; k < 6; k++) {
            t = gf_fix_add(t, gf_fix_split(x[k], elow));
            v = v + x[k];
        }
        volatile double q = v / 6.0;
        const double want = q, got = gf_fix_ok(t) ? gf_fix_div6(t, elow) : want;
        n++;
        bad += memcmp(&want, &got, 8) != 0;
    }
    printf("div6 checked %lld mismatches %lld, highest window %u\n", n, bad, (unsigned)GF_FIX_TOP);
    return 0;
}
