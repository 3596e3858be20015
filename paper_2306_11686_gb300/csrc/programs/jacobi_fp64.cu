/*
 * The Jacobi program's second kernel: the sweeps on the FP64 pipe, at 4
 * resident blocks per SM (jacobi.cu says what takes it here).
 */
#include <stdlib.h>
#include "jacobi.cuh"

/*
 * The same sweep written with the k loop inside the parallel loop: work item
 * t is the column (i, j) over planes [k0, k0 + kseg), t = (k0 / kseg) * n^2 +
 * j * n + i, so consecutive items are consecutive i (coalesced).  Walking up
 * the column, the k - 1 and k neighbours of a point are the values loaded for
 * the previous point, so each point loads five values instead of seven, and
 * the index split and boundary test are paid once per column segment.  Every
 * point's arithmetic and its order are those of jacobi_sweep, so the grid
 * and the residual are the same bits.
 */
template <int INT_ADDS>
__device__ int jacobi_sweep_col(const double *u, double *un, uint32_t nn, gf_udiv32 dn, gf_udiv32 dsk, uint32_t kseg,
                                double *res)
{
    const uint32_t sk = nn * nn;
    const uint32_t nseg = (nn + kseg - 1) / kseg;
    return gf_reduce<double, GF_RED_MAX>(
        0, (int64_t)nseg * sk, GF_SCHED_STATIC, 1,
        [=](int64_t t64) -> double {
            const uint32_t t = (uint32_t)t64;
            const uint32_t seg = dsk.div(t), ij = t - seg * sk;
            const uint32_t j = dn.div(ij), im1 = ij - 1u - j * nn;
            const uint32_t k0 = seg * kseg, k1 = min(k0 + kseg, nn);
            double *o = un + ij;
            if (max(im1, j - 1u) >= nn - 2u) {            /* a boundary column */
                for (uint32_t k = k0; k < k1; k++)
                    o[(size_t)k * sk] = 0.0;
                return 0.0;
            }
            const double *c = u + ij;
            uint32_t k = k0;
            if (k == 0) {                                  /* the bottom boundary plane */
                o[0] = 0.0;
                k = 1;
            }
            const uint32_t kend = min(k1, nn - 1u);
            long long best = 0;                            /* bits of the largest |un - u|, +0 to start */
            if (k < kend) {
                double um = __ldg(c + (size_t)(k - 1) * sk), u0 = __ldg(c + (size_t)k * sk);
                for (; k < kend; k++) {
                    const double *p = c + (size_t)k * sk;
                    const double up = __ldg(p + sk);
                    const double nb[6] = {__ldg(p - 1), __ldg(p + 1), __ldg(p - nn), __ldg(p + nn), um, up};
                    double v = nb[0];
#pragma unroll
                    for (int q = 1; q < 6; q++)
                        v = q <= INT_ADDS ? gf_dadd_int(v, nb[q]) : __dadd_rn(v, nb[q]);
                    v = gf_div6_int(v);
                    o[(size_t)k * sk] = v;
                    /* |un - u| >= 0: its bits order as the values do; NaN is skipped, as the reduction does */
                    const long long b = __double_as_longlong(gf_fabs_int(__dadd_rn(v, -u0)));
                    if (b <= 0x7ff0000000000000ll && b > best)
                        best = b;
                    um = u0;
                    u0 = up;
                }
            }
            if (k1 == nn && nn > 1)                        /* the top boundary plane */
                o[(size_t)(nn - 1) * sk] = 0.0;
            return __longlong_as_double(best);
        },
        res);
}

/* options: this kernel's sweeps; grids for which the first kernel looks for a window may need both */
static int jacobi_pick(int argc, const char *const *argv)
{
    if (argc > 4)
        return GF_SECOND_ONLY;
    const long long n = argc > 1 ? atoll(argv[1]) : 0;
    return n > 0 && n <= 1290 && n * n * n >= (long long)JACOBI_FIX_CELLS ? GF_BOTH : GF_FIRST_ONLY;
}

GF_SECOND(jacobi, jacobi_fp64, 4, jacobi_pick)(int argc, char **argv)
{
    jacobi_job job;
    if (!jacobi_parse(argc, argv, &job))
        return 2;
    double *owned = nullptr;
    int s = 1;
    if (gfd::s_st->second == 2u) {                 /* from sweep s on, with the first kernel's grid */
        s = (int)gfd::s_st->second_arg[0];
        owned = (double *)gfd::s_st->second_arg[1];
    }
    /* the index split's magic numbers: loop invariants, made once */
    const uint32_t nn = job.nn, ks = (uint32_t)job.kseg;
    const gf_udiv32 dn = gf_udiv32::make(nn), dsk = gf_udiv32::make(nn * nn);
    for (; s <= job.sweeps; s++) {
        const double *u = owned ? owned : job.u0;
        double *un = jacobi_grid(job, s), res = 0.0;
        if (!un)
            return 4;
        int rc;
        if (ks > 0) {
            switch (job.int_adds) {
            case 0: rc = jacobi_sweep_col<0>(u, un, nn, dn, dsk, ks, &res); break;
            case 1: rc = jacobi_sweep_col<1>(u, un, nn, dn, dsk, ks, &res); break;
            case 2: rc = jacobi_sweep_col<2>(u, un, nn, dn, dsk, ks, &res); break;
            case 3: rc = jacobi_sweep_col<3>(u, un, nn, dn, dsk, ks, &res); break;
            case 4: rc = jacobi_sweep_col<4>(u, un, nn, dn, dsk, ks, &res); break;
            default: rc = jacobi_sweep_col<5>(u, un, nn, dn, dsk, ks, &res); break;
            }
        } else {
            switch (job.int_adds) {
            case 0: rc = jacobi_sweep<0>(u, un, nn, dn, job.cells, &res); break;
            case 1: rc = jacobi_sweep<1>(u, un, nn, dn, job.cells, &res); break;
            case 2: rc = jacobi_sweep<2>(u, un, nn, dn, job.cells, &res); break;
            case 3: rc = jacobi_sweep<3>(u, un, nn, dn, job.cells, &res); break;
            case 4: rc = jacobi_sweep<4>(u, un, nn, dn, job.cells, &res); break;
            default: rc = jacobi_sweep<5>(u, un, nn, dn, job.cells, &res); break;
            }
        }
        if (rc)
            return 10;
        jacobi_swap(s, res, un, &owned);
    }
    return jacobi_write(job, owned);
}
