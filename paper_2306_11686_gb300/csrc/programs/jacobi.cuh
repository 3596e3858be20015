/*
 * What the two kernels of the Jacobi program share: its arguments, the sweep
 * with one parallel iteration per point, and the end of the program.
 */
#ifndef GF_JACOBI_CUH
#define GF_JACOBI_CUH
#include "../gf_device.cuh"
#include "../gf_fastdiv.cuh"
#include "../gf_intpipe.cuh"

/* grids from here on: a sweep of 96^3 takes 18.0 us on either path, of 112^3 16.9 against 24.7 us; smaller ones
 * would also pay for the sample's two regions (10 us) */
#define JACOBI_FIX_CELLS (1u << 20)

struct jacobi_job {
    uint32_t nn;
    int sweeps, int_adds;
    long long kseg;
    uint64_t cells;
    const double *u0;              /* the input grid */
    const char *path;
};

/* jacobi n sweeps out_path [int_adds [kseg]]: false for arguments that the program refuses */
static __device__ bool jacobi_parse(int argc, char **argv, jacobi_job *job)
{
    if (argc < 4)
        return false;
    const long long n = gf_atoll(argv[1]);
    job->sweeps = (int)gf_atoll(argv[2]);
    job->path = argv[3];
    job->int_adds = argc > 4 ? (int)gf_atoll(argv[4]) : 1;
    job->kseg = argc > 5 ? gf_atoll(argv[5]) : 0;
    job->u0 = (const double *)gf_buffer(0);
    job->cells = (uint64_t)n * n * n;
    job->nn = (uint32_t)n;
    return n >= 1 && n <= 1290 && job->u0 && gf_buffer_bytes(0) >= job->cells * 8 && job->int_adds >= 0 &&
           job->int_adds <= 5 && job->kseg >= 0 && job->kseg <= n;
}

/* a sweep's new grid; the program ends without one */
static __device__ double *jacobi_grid(const jacobi_job &job, int s)
{
    double *un = (double *)gf_malloc(job.cells * sizeof(double));
    if (!un)
        gf_printf("jacobi: out of device heap at sweep %d\n", s);
    return un;
}

/* the sweep's line, and the grid before goes; the new one is *owned */
static __device__ void jacobi_swap(int s, double res, double *un, double **owned)
{
    gf_printf("%d %.17g\n", s, res);
    if (*owned)
        gf_free(*owned);
    *owned = un;
}

/* the last grid to the file ("-": write nothing, for profiling); the exit code */
static __device__ int jacobi_write(const jacobi_job &job, double *owned)
{
    const double *u = owned ? owned : job.u0;
    size_t w = job.cells;
    if (job.path[0] != '-' || job.path[1] != 0) {
        GF_FILE f = gf_fopen(job.path, "wb");
        if (!f)
            return 3;
        w = gf_fwrite(u, sizeof(double), (size_t)job.cells, f);
        gf_fclose(f);
    }
    if (owned)
        gf_free(owned);
    return w == job.cells ? 0 : 3;
}

/*
 * One Jacobi sweep: the six-neighbour average of the interior into un, 0 on
 * the boundary, and the max residual |un - u| over the grid as a max
 * reduction.  The five neighbour adds keep the serial program's order; the
 * first INT_ADDS of them run on the integer pipe and the rest on the FP64
 * pipe (every one correctly rounded, so the split changes no bit of the
 * result, only which pipe does the work), as do the division by 6 and the
 * absolute value.  The flat index is split into (i, j, k) by multiplication
 * with an invariant-divisor magic number.
 */
template <int INT_ADDS>
__device__ int jacobi_sweep(const double *u, double *un, uint32_t nn, gf_udiv32 dn, uint64_t cells, double *res)
{
    const uint32_t sk = nn * nn;
    return gf_reduce<double, GF_RED_MAX>(
        0, (int64_t)cells, GF_SCHED_STATIC, 1,
        [=](int64_t c64) -> double {
            const uint32_t c = (uint32_t)c64;
            /* i - 1, j - 1, k - 1 wrap to 2^32 - 1 at 0, so one unsigned
             * compare of their maximum finds every boundary cell */
            const uint32_t jk = dn.div(c), im1 = c - 1u - jk * nn;
            const uint32_t k = dn.div(jk), jm1 = jk - 1u - k * nn;
            if (max(im1, max(jm1, k - 1u)) >= nn - 2u) {
                un[c] = 0.0;
                return 0.0;
            }
            /* u is not written during the sweep: read-only loads, which may be
             * issued ahead of the previous iteration's store to un */
            const double nb[6] = {__ldg(u + c - 1),  __ldg(u + c + 1),  __ldg(u + c - nn),
                                  __ldg(u + c + nn), __ldg(u + c - sk), __ldg(u + c + sk)};
            double v = nb[0];
#pragma unroll
            for (int t = 1; t < 6; t++)
                v = t <= INT_ADDS ? gf_dadd_int(v, nb[t]) : __dadd_rn(v, nb[t]);
            v = gf_div6_int(v);               /* == v / 6.0, bit for bit */
            un[c] = v;
            return gf_fabs_int(__dadd_rn(v, -__ldg(u + c)));
        },
        res);
}

#endif
