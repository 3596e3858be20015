/* Host check of gf_fixsum.cuh: six values of +0 are a sum that is accepted,
 * and its sixth is +0, in every window; with one -0 they are not accepted.
 *
 *   fixsum_zero_check      prints "zero checked N mismatches M" */
#include <cstdio>
#include "gf_fixsum.cuh"

int main()
{
    long long n = 0, bad = 0;
    for (uint32_t elow = 5; elow + 8u <= GF_FIX_TOP; elow++)
        for (int minus = -1; minus < 6; minus++) {
            gf_fix3 t = gf_fix_split(minus == 0 ? -0.0 : 0.0, elow);
            for (int k = 1; k < 6; k++)
                t = gf_fix_add(t, gf_fix_split(minus == k ? -0.0 : 0.0, elow));
            n++;
            bad += minus < 0 ? !gf_fix_ok(t) || gf_ip_bits(gf_fix_div6(t, elow)) != 0u : gf_fix_ok(t);
        }
    printf("zero checked %lld mismatches %lld\n", n, bad);
    return bad != 0;
}
