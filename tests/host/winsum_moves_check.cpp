/* Host check of how often gf_winsum.cuh gives work to the FP64 sum: warps of
 * 32 threads add values side by side, and every step costs the warp what its
 * busiest lane adds (the others wait).  Without windows that is one addition
 * a step.
 *
 *   winsum_moves_check          prints "KIND adds A steps S" for each kind of data */
#include <cmath>
#include <cstdio>
#include "gf_winsum.cuh"

static uint64_t s_rng = 3;
static uint64_t rnd()
{
    uint64_t z = (s_rng += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double unit() { return 0.5 + (double)(rnd() >> 12) * 0x1p-53; }      /* [0.5, 1) */

static void run(const char *name, double (*value)(int step))
{
    const int steps = 216, warps = 64;
    long long adds = 0;
    for (int w = 0; w < warps; w++) {
        gf_winsum t[32];
        uint32_t room[32];
        for (uint32_t &r : room)
            r = GF_WIN_TERMS;
        for (int s = 0; s < steps; s++) {
            int most = 0;
            for (int l = 0; l < 32; l++) {
                int n = 0;
                auto add = [&](double) { n++; };
                const double x = value(s);
                const uint32_t p = t[l].place(x);
                if (p <= 31u && t[l].base) {
                    t[l].add_in(x, p);
                    if (--room[l] == 0u) {
                        t[l].fold(add);
                        room[l] = GF_WIN_TERMS;
                    }
                } else {
                    t[l].add_out(x, add, room[l]);
                }
                most = n > most ? n : most;
            }
            adds += most;
        }
    }
    printf("%s adds %lld steps %lld\n", name, adds, (long long)steps * warps);
}

template <int SPREAD> static double spread(int) { return ldexp(unit(), (int)(rnd() % SPREAD) - SPREAD / 2); }

int main()
{
    run("uniform", [](int) { return (double)(rnd() >> 11) * 0x1p-53; });
    run("spread40", spread<40>);
    run("spread64", spread<64>);
    run("spread128", spread<128>);
    run("spread600", spread<600>);
    run("fifth", [](int) { return rnd() % 5 ? unit() : unit() * 0x1p-60; });
    run("drift", [](int s) { return ldexp(unit(), s / 4); });
    return 0;
}
