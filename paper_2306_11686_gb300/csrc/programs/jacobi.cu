/*
 * The Laplace Jacobi program (the benchmark): a legacy stencil code run whole
 * on the GPU -- per-sweep malloc/free, a max reduction and a printf, the final
 * grid written to a file.  Its serial twin in plain C with the real libc is
 * what a run must reproduce, bit for bit.
 */
#include "jacobi.cuh"
#include "../gf_fixsum.cuh"

/*
 * The sweep for the grids that no fixed-point window suits, in the kernel that
 * is compiled for the fixed-point sweep (2 blocks per SM): columns of
 * JACOBI_SEG planes, every add on the FP64 pipe, and the loads of the next
 * point on their way while one is computed, because 16 warps an SM do not hide
 * them.  256^3 with values of both signs: 204 us (jacobi_sweep<0> 212 here;
 * the FP64 pipe's six operations a point alone take 186); segments of 2, 4, 8
 * and 16 planes 203.8, 204.2, 204.6 and 209.3; two points at a time 217; the
 * first add on the integer pipe 205 to 233.
 */
#define JACOBI_SEG 4u
static __device__ int jacobi_sweep_ahead(const double *u, double *un, uint32_t nn, gf_udiv32 dn, gf_udiv32 dsk,
                                         double *res)
{
    const uint32_t sk = nn * nn;
    return gf_reduce<double, GF_RED_MAX>(
        0, (int64_t)((nn + JACOBI_SEG - 1u) / JACOBI_SEG) * sk, GF_SCHED_STATIC, 1,
        [=](int64_t t64) -> double {
            const uint32_t t = (uint32_t)t64;
            const uint32_t seg = dsk.div(t), ij = t - seg * sk;
            const uint32_t j = dn.div(ij), im1 = ij - 1u - j * nn;
            const uint32_t k0 = seg * JACOBI_SEG, k1 = min(k0 + JACOBI_SEG, nn);
            double *o = un + ij;
            if (max(im1, j - 1u) >= nn - 2u) {            /* a boundary column */
                for (uint32_t k = k0; k < k1; k++)
                    o[(size_t)k * sk] = 0.0;
                return 0.0;
            }
            uint32_t k = k0;
            if (k == 0) {                                  /* the bottom boundary plane */
                o[0] = 0.0;
                k = 1;
            }
            const uint32_t kend = min(k1, nn - 1u);
            long long best = 0;                            /* bits of the largest |un - u|, +0 to start */
            if (k < kend) {
                const double *p = u + ij + (size_t)k * sk;
                o += (size_t)k * sk;
                double um = __ldg(p - sk), u0 = __ldg(p);
                double il = __ldg(p - 1), ir = __ldg(p + 1), jl = __ldg(p - nn), jr = __ldg(p + nn), up = __ldg(p + sk);
                for (;;) {
                    double il1, ir1, jl1, jr1, up1;
                    const bool more = ++k < kend;
                    if (more) {
                        p += sk;
                        il1 = __ldg(p - 1), ir1 = __ldg(p + 1), jl1 = __ldg(p - nn), jr1 = __ldg(p + nn);
                        up1 = __ldg(p + sk);
                    }
                    double v = __dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(il, ir), jl), jr), um), up);
                    v = gf_div6_int(v);
                    *o = v;
                    /* |un - u| >= 0: its bits order as the values do; NaN is skipped, as the reduction does */
                    const long long b = __double_as_longlong(gf_fabs_int(__dadd_rn(v, -u0)));
                    if (b <= 0x7ff0000000000000ll && b > best)
                        best = b;
                    if (!more)
                        break;
                    o += sk;
                    um = u0, u0 = up, up = up1, il = il1, ir = ir1, jl = jl1, jr = jr1;
                }
            }
            if (k1 == nn && nn > 1)                        /* the top boundary plane */
                un[ij + (size_t)(nn - 1) * sk] = 0.0;
            return __longlong_as_double(best);
        },
        res);
}

/* What a fixed-point sweep reduces: the largest |un - u| (its bits, NaN left
 * out), the largest high word among the old values of the planes that could
 * raise it (a sample, from which the next sweep's window is taken) and the
 * number of points left out. */
struct jacobi_red {
    unsigned long long res;
    int hi;
    uint32_t out;
};
namespace gfd {
template <> struct acc<jacobi_red, GF_RED_MAX> {
    jacobi_red v;
    __device__ acc() : v{0ull, 0, 0u} {}
    __device__ void add(const jacobi_red &x)
    {
        v.res = x.res > v.res ? x.res : v.res;
        v.hi = x.hi > v.hi ? x.hi : v.hi;
        v.out += x.out;
    }
    __device__ void merge(const acc &o) { add(o.v); }
    __device__ jacobi_red result() const { return v; }
    __device__ void to_words(uint64_t *w) const
    {
        w[0] = v.res;
        w[1] = (uint64_t)(uint32_t)v.hi << 32 | v.out;
    }
    __device__ void from_words(const uint64_t *w)
    {
        v.res = w[0];
        v.hi = (int)(w[1] >> 32);
        v.out = (uint32_t)w[1];
    }
    __device__ acc shfl_xor(int m) const
    {
        acc r;
        r.v.res = __shfl_xor_sync(0xffffffffu, v.res, m);
        r.v.hi = __shfl_xor_sync(0xffffffffu, v.hi, m);
        r.v.out = __shfl_xor_sync(0xffffffffu, v.out, m);
        return r;
    }
};
} // namespace gfd

/* a point the fixed-point sweep leaves out: the serial program's operations */
static __device__ __noinline__ double jacobi_point(const double *p, uint32_t nn, uint32_t sk)
{
    double v = __dadd_rn(__ldg(p - 1), __ldg(p + 1));
    v = __dadd_rn(v, __ldg(p - nn));
    v = __dadd_rn(v, __ldg(p + nn));
    v = __dadd_rn(v, __ldg(p - (size_t)sk));
    v = __dadd_rn(v, __ldg(p + (size_t)sk));
    return v / 6.0;
}

#define JACOBI_ROWS 4        /* rows of a lane */
#define JACOBI_OUT 30u       /* points of a warp's row that it writes */
#define JACOBI_AHEAD 2       /* planes on their way ahead of the one being computed */
#define JACOBI_SLOT ((JACOBI_ROWS + 2) * 256u)              /* bytes of a plane's rows in a warp's ring */
#define JACOBI_LEFT 0x7ff4a5a55a5a5a5aull   /* marks a point left to the FP64 path (computing it again is always right) */

__shared__ double s_jacobi_ring[GF_MAX_WARPS][(JACOBI_AHEAD + 1) * (JACOBI_ROWS + 2) * 32];

__device__ __forceinline__ void copy8_async(uint32_t dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ double lds_f64(uint32_t a)
{
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

/* the point at p / o, if a fixed-point sweep left it out */
static __device__ __forceinline__ void jacobi_left(const double *p, double *o, uint32_t nn, uint32_t sk, jacobi_red *r)
{
    if (gf_ip_bits(*o) != JACOBI_LEFT)
        return;
    const double v = jacobi_point(p, nn, sk);
    *o = v;
    const unsigned long long b = gf_ip_bits(__dadd_rn(v, -__ldg(p))) & 0x7fffffffffffffffull;
    r->res = b <= 0x7ff0000000000000ull && b > r->res ? b : r->res;
    r->hi = max(r->hi, (int)(gf_ip_bits(v) >> 32));
}

/* every point that a fixed-point sweep left out, by the whole grid */
static __device__ int jacobi_rest(const double *u, double *un, uint32_t nn, uint32_t cells, jacobi_red *red)
{
    const uint32_t sk = nn * nn;
    return gf_reduce<jacobi_red, GF_RED_MAX>(
        0, (int64_t)cells, GF_SCHED_STATIC, 1,
        [=](int64_t c) -> jacobi_red {
            jacobi_red r{0ull, 0, 0u};
            jacobi_left(u + c, un + c, nn, sk, &r);
            return r;
        },
        red);
}

/* how a fixed-point sweep cuts the grid: `tiles` columns of a warp each, in `segs` segments of `len` planes;
 * warps x 32 parallel iterations take the tiles x segs items round robin */
struct jacobi_cut {
    uint32_t tiles, segs, len, warps;
};

/*
 * The same sweep on the FP32 pipe (gf_fixsum.cuh): the adds and the division
 * round as the serial program's, so grid and residual are the same bits.
 *
 * A warp's 32 lanes are 32 consecutive points of a band of rows, of which the
 * inner 30 are written; each lane walks up k with JACOBI_ROWS rows of j.  A
 * point's chunks are made once and serve as its own row's k - 1 and k + 1
 * neighbours and the next rows' j neighbours (registers) and as the i
 * neighbours of the lanes beside it (shuffles); only the two rows just
 * outside the band are converted again by the next band.  Each lane copies
 * its own rows of the planes ahead into a ring in shared memory (cp.async:
 * no registers held while they fly, and no other thread reads them).
 *
 * The residual's maximum costs little: a plane whose residuals all lie below
 * the warp's own maximum so far (by their high words) is done, any other goes
 * through the exact maximum.
 *
 * What bounds it: issue slots and the integer pipe (142 warp instructions per
 * 30 points, 58 of them integer; 69% of the issue slots and 56% of the integer
 * pipe busy, 0.24 GB of DRAM traffic a sweep).  A sweep of 256^3 takes 104 us
 * (102.5 if sums of zeros were left out) against 173 us for jacobi_sweep<1> at 4 blocks per SM (the FP64 pipe's 5
 * operations a point alone take 155 us).  Measured for this layout in a kernel
 * of its own, us: rows 2 / 3 / 4 / 5 / 6 at the best of 2 to 4 blocks per SM
 * 98 / 94 / 91 / 90 / 92; in the program 4 rows at 2 blocks per SM lead (104
 * against 114 for 3 rows at 3 and 111 for 5 at 2).  Loads straight into
 * registers one plane ahead 137; whole columns of 256 planes 160 (neighbour
 * bands drift apart and DRAM reads grow 2.7x); one row of four on the FP64
 * pipe 118 (its latency shows).
 */
struct jacobi_fix_body {
    const double *u;
    double *un;
    uint32_t nn, elow;
    gf_udiv32 dn, dt;
    jacobi_cut cut;
    __device__ __forceinline__ jacobi_red operator()(int64_t t64) const
    {
        const uint32_t sk = nn * nn;
        const uint32_t nf = (nn + JACOBI_ROWS - 1u) / JACOBI_ROWS * nn;      /* points of all bands' first rows */
        constexpr int R = JACOBI_ROWS;
        const uint32_t lane = (uint32_t)t64 & 31u, wid = (uint32_t)(t64 >> 5);
        const uint32_t ring =
            (uint32_t)__cvta_generic_to_shared(&s_jacobi_ring[threadIdx.x >> 5][threadIdx.x & 31u]);
        jacobi_red r{0ull, 0, 0u};
        uint32_t top = 0u;                             /* high word of the warp's largest residual */
        /* consecutive items go to consecutive blocks, so that a last round that is not full is spread over the SMs */
        for (uint32_t item = (wid & 7u) * (cut.warps >> 3) + (wid >> 3); item < cut.tiles * cut.segs;
             item += cut.warps) {
            const uint32_t seg = dt.div(item), tile = item - seg * cut.tiles;
            const uint32_t k0 = seg * cut.len, k1 = min(k0 + cut.len, nn);
            const uint32_t f0 = tile * JACOBI_OUT + lane;                    /* one past the point's index */
            const bool mine = lane - 1u < JACOBI_OUT && f0 - 1u < nf;
            const uint32_t f = f0 == 0u ? 0u : min(f0 - 1u, nf - 1u);
            const uint32_t jb = dn.div(f), i = f - jb * nn, j0 = jb * R;
            uint32_t off[R];                           /* the rows, clamped into the grid (a clamped row's values are not used) */
            uint32_t wr = 0u, in = 0u;                 /* this lane's points, a bit a row; of them the interior ones */
#pragma unroll
            for (int q = 0; q < R; q++) {
                off[q] = min(j0 + q, nn - 1u) * nn + i;
                const bool w = mine && j0 + q < nn;
                wr |= w ? 1u << q : 0u;
                in |= w && i - 1u < nn - 2u && j0 + q - 1u < nn - 2u ? 1u << q : 0u;
            }
            const uint32_t offa = j0 ? off[0] - nn : off[0], offd = min(j0 + R, nn - 1u) * nn + i;
            if (wr != in || k0 == 0 || k1 == nn)       /* boundary points */
                for (uint32_t k = k0; k < k1; k++)
#pragma unroll
                    for (int q = 0; q < R; q++)
                        if ((wr >> q & 1u) && (!(in >> q & 1u) || k - 1u >= nn - 2u))
                            un[(size_t)k * sk + off[q]] = 0.0;
            uint32_t k = k0 ? k0 : 1u;
            const uint32_t kend = min(k1, nn - 1u);
            if (k >= kend)
                continue;
            const double *p = u + (size_t)k * sk;
            double *o = un + (size_t)k * sk;
            uint32_t left0 = 0u, left1 = 0u, left = 0u;     /* first and last plane with points left out, this lane's count */
            gf_fix3 m[R], c[R], s[R];                  /* planes k - 1 and k in chunks; the sums */
            /* a ring slot holds the centre rows of a plane and the halo rows of the plane below it */
            auto fetch = [&](uint32_t slot, const double *pl, bool halo) {
#pragma unroll
                for (int q = 0; q < R; q++)
                    copy8_async(slot + q * 256u, pl + off[q]);
                if (halo) {
                    copy8_async(slot + R * 256u, pl + ((int)offa - (int)sk));
                    copy8_async(slot + (R + 1) * 256u, pl + ((int)offd - (int)sk));
                }
            };
            fetch(ring, p, false);
            fetch(ring + JACOBI_SLOT, p + sk, true);
            copy_commit();
            const double *ahead = p + 2 * (size_t)sk;  /* the next plane to fetch, up to kend */
#pragma unroll
            for (int d = 2; d <= JACOBI_AHEAD; d++) {
                if (k + d <= kend)
                    fetch(ring + d * JACOBI_SLOT, ahead, true);
                copy_commit();
                ahead += sk;
            }
#pragma unroll
            for (int q = 0; q < R; q++)
                m[q] = gf_fix_split(__ldg(p - sk + off[q]), elow);
            copy_wait<JACOBI_AHEAD - 1>();
#pragma unroll
            for (int q = 0; q < R; q++)
                c[q] = gf_fix_split(lds_f64(ring + q * 256u), elow);
            uint32_t here = ring, next = ring + JACOBI_SLOT;      /* slots of planes k and k + 1 */
#pragma unroll 2
            for (; k < kend; k++) {
                copy_wait<JACOBI_AHEAD - 1>();
#pragma unroll
                for (int q = 0; q < R; q++) {          /* i - 1 and i + 1 */
                    gf_fix3 l, g;
                    l.a = __shfl_up_sync(0xffffffffu, c[q].a, 1);
                    l.b = __shfl_up_sync(0xffffffffu, c[q].b, 1);
                    l.c = __shfl_up_sync(0xffffffffu, c[q].c, 1);
                    g.a = __shfl_down_sync(0xffffffffu, c[q].a, 1);
                    g.b = __shfl_down_sync(0xffffffffu, c[q].b, 1);
                    g.c = __shfl_down_sync(0xffffffffu, c[q].c, 1);
                    s[q] = gf_fix_add(l, g);
                }
                {                                      /* j - 1, j + 1 and k - 1 */
                    const gf_fix3 a = gf_fix_split(lds_f64(next + R * 256u), elow);
                    const gf_fix3 d = gf_fix_split(lds_f64(next + (R + 1) * 256u), elow);
#pragma unroll
                    for (int q = 0; q < R; q++) {
                        s[q] = gf_fix_add(s[q], q ? c[q - 1] : a);
                        s[q] = gf_fix_add(s[q], q < R - 1 ? c[q + 1] : d);
                        s[q] = gf_fix_add(s[q], m[q]);
                    }
                }
                uint32_t bh[R], bl[R], big = 0u;       /* the residuals' bits */
                float least = 1.0f;                    /* NaN: a sum was not computed here */
#pragma unroll
                for (int q = 0; q < R; q++) {
                    m[q] = c[q];
                    c[q] = gf_fix_split(lds_f64(next + q * 256u), elow);
                    s[q] = gf_fix_add(s[q], c[q]);     /* k + 1 */
                    const double v = gf_fix_div6(s[q], elow);
                    if (in & (1u << q))
                        o[off[q]] = v;
                    const uint64_t b = gf_ip_bits(__dadd_rn(v, -lds_f64(here + q * 256u)));
                    bl[q] = (uint32_t)b;
                    bh[q] = (uint32_t)(b >> 32) & 0x7fffffffu;
                    big = max(big, bh[q]);
                    asm("min.NaN.f32 %0, %0, %1;" : "+f"(least) : "f"(s[q].a));
                }
                if (__any_sync(0xffffffffu, in != 0u && (big >= top || !(least >= 0.0f)))) {
                    big = top;
                    const uint32_t before = left;
#pragma unroll
                    for (int q = 0; q < R; q++) {
                        if (!(in & (1u << q)))
                            continue;
                        if (!gf_fix_ok(s[q]) || bh[q] >= 0x7ff00000u) {   /* outside the window, or no finite residual */
                            o[off[q]] = __longlong_as_double((long long)JACOBI_LEFT);
                            left++;
                        } else {
                            const unsigned long long b = (uint64_t)bh[q] << 32 | bl[q];
                            r.res = b > r.res ? b : r.res;
                            big = max(big, bh[q]);
                        }
                        r.hi = max(r.hi, (int)(gf_ip_bits(lds_f64(here + q * 256u)) >> 32));
                    }
                    top = __reduce_max_sync(0xffffffffu, big);
                    if (__any_sync(0xffffffffu, left != before)) {
                        left0 = left0 ? left0 : k;
                        left1 = k;
                    }
                }
                if (k + (JACOBI_AHEAD + 1) <= kend)    /* into the slot of plane k, which is done */
                    fetch(here, ahead, true);
                copy_commit();
                ahead += sk;
                o += sk;
                here = next;
                next += JACOBI_SLOT;
                next = next == ring + (JACOBI_AHEAD + 1) * JACOBI_SLOT ? ring : next;
            }
            copy_wait<0>();
            if (left0 == 0u || left1 - left0 > 3u) {   /* many: the caller runs jacobi_rest */
                r.out += left;
                continue;
            }
            for (k = left0; k <= left1; k++)           /* few (a corner of the grid, say): here */
#pragma unroll 1
                for (uint32_t q = 0; q < (uint32_t)R; q++) {
                    const size_t to = (size_t)k * sk + min(j0 + q, nn - 1u) * nn + i;
                    if (left && (in >> q & 1u))
                        jacobi_left(u + to, un + to, nn, sk, &r);
                }
        }
        return r;
    }
};

#define JACOBI_SAMPLE 32768
/* a sample of the grid's values.  elow = 0: their largest high word, in red->out how many no window can hold
 * (negative, infinite, NaN or above the highest) and, 2^16 each, how many are zero; else in red->out how many lie
 * outside the window that starts at elow */
static __device__ int jacobi_sample(const double *u, uint32_t cells, uint32_t elow, jacobi_red *red)
{
    return gf_reduce<jacobi_red, GF_RED_MAX>(
        0, JACOBI_SAMPLE, GF_SCHED_STATIC, 1,
        [=](int64_t t) -> jacobi_red {
            uint32_t h = (uint32_t)t * 0x9E3779B1u;            /* spread over the grid: no plane or row alone */
            h ^= h >> 15;
            h *= 0x85EBCA6Bu;
            h ^= h >> 13;
            const uint64_t b = gf_ip_bits(__ldg(u + __umulhi(h, cells)));
            const uint32_t hi = (uint32_t)(b >> 32);
            if (elow == 0u)
                return jacobi_red{0ull, (int)hi, (hi >> 20 > GF_FIX_TOP ? 1u : 0u) + (b << 1 == 0ull ? 0x10000u : 0u)};
            return jacobi_red{0ull, (int)hi, b != 0ull && (hi >> 20) - elow > 8u ? 1u : 0u};
        },
        red);
}

/* the lowest binade (biased exponent) of the fixed-point window that suits the grid u, 0 if none does: less
 * than one value in 4096 may lie outside it (each costs up to six points the FP64 path).  +0 lies in every
 * window; a sample of nothing else takes the one that ends at 2, and the first sweep sees what there is.
 * *fp64: the second kernel is the faster one for the grid, because the values outside have not halved since the
 * last sample (*outside; values that are spread at random fall into a window within a few sweeps, smooth or signed
 * ones do not); a grid with many zeros gains nothing there. */
static __device__ uint32_t jacobi_window(const double *u, uint32_t cells, uint32_t *outside, bool *fp64, int *rc)
{
    jacobi_red red{0ull, 0, 0u};
    *rc = jacobi_sample(u, cells, 0u, &red);
    const uint32_t top = (uint32_t)red.hi >> 20, zeros = red.out >> 16, before = *outside;
    uint32_t bad = red.out & 0xffffu;
    *fp64 = false;
    if (!*rc && zeros == JACOBI_SAMPLE && bad == 0u)
        return 1015u;
    if (!*rc && bad <= JACOBI_SAMPLE / 4096 && top >= 13u && top <= GF_FIX_TOP) {
        *rc = jacobi_sample(u, cells, top - 8u, &red);
        bad = red.out;
        if (!*rc && bad <= JACOBI_SAMPLE / 4096)
            return top - 8u;
    }
    *outside = bad;
    *fp64 = zeros <= JACOBI_SAMPLE / 8 && 2u * bad > before;
    return 0u;
}

/* segments of k for the fixed-point sweep: with r rounds of the warps' items there is room for r * warps / tiles
 * segments; the longest walk is then r * (len + 1.5) planes (a segment's start costs about 1.5) */
static __device__ jacobi_cut jacobi_make_cut(uint32_t nn, uint32_t warps)
{
    jacobi_cut c{(((nn + JACOBI_ROWS - 1u) / JACOBI_ROWS) * nn + JACOBI_OUT - 1u) / JACOBI_OUT, 1u, nn,
                 max(8u, warps & ~7u)};
    const uint32_t r0 = (c.tiles + c.warps - 1u) / c.warps;
    uint32_t least = 0xffffffffu;
    for (uint32_t r = r0; r < r0 + 6u; r++) {
        const uint32_t len = max(2u, (nn * c.tiles + r * c.warps - 1u) / (r * c.warps));      /* ceil(nn / (r warps / tiles)) */
        const uint32_t segs = (nn + len - 1u) / len;
        const uint32_t cost = (segs * c.tiles + c.warps - 1u) / c.warps * (2u * len + 3u);
        if (cost < least) {
            least = cost;
            c.segs = segs;
            c.len = len;
        }
    }
    return c;
}

/*
 * jacobi n sweeps out_path [int_adds [kseg]]   buffers: 0 = input grid (n^3 doubles, i fastest)
 *
 * Laplace Jacobi sweeps with the six-neighbour average, boundary written as 0,
 * a fresh grid from the device heap every sweep (old one freed after the
 * swap), the max residual over the interior fused into the sweep as a max
 * reduction, one printf per sweep, the final grid fwrite'd.  Without further
 * arguments a sweep runs on the FP32 pipe (jacobi_fix_body) while a window
 * of binades holds the grid's values, else on the FP64 pipe.  int_adds (0..5)
 * asks for jacobi_sweep with that many of the five neighbour adds on the
 * integer pipe; kseg > 0 runs it as columns of kseg planes
 * (jacobi_sweep_col) instead of one parallel iteration per point.
 *
 * Two kernels: jacobi_fix_body wants 104 registers, 2 resident blocks per SM,
 * and the FP64-pipe sweeps want 4 (256^3, uniform data: 173 us with one
 * integer add at 4 blocks per SM, 217 at 2).  The first kernel has the
 * fixed-point sweep, and FP64 sweeps for small grids, for the time between two
 * samples and for grids with many zeros.  The second one has the sweeps that
 * the options ask for, and takes over the grids that no window will suit.
 */
/* The fixed sweep is part of the worker loop: behind the trampoline pointer it took 111 us. */
using jacobi_hot = gfd::hot_reduce<jacobi_red, GF_RED_MAX, jacobi_fix_body>;
GF_MAIN_HOT(jacobi, 2, jacobi_hot)(int argc, char **argv)
{
    jacobi_job job;
    if (!jacobi_parse(argc, argv, &job))
        return 2;
    double *owned = nullptr;
    const uint32_t nn = job.nn, cells = (uint32_t)job.cells;
    /* the index split's magic numbers: loop invariants, made once */
    const gf_udiv32 dn = gf_udiv32::make(nn), dsk = gf_udiv32::make(nn * nn);
    const jacobi_cut cut = jacobi_make_cut(nn, (uint32_t)(gfd::s_st->nworkers >> 5));
    const gf_udiv32 dt = gf_udiv32::make(cut.tiles);
    uint32_t elow = 0u;                            /* window of the fixed-point sweeps, 0: not known */
    int ask = 0, pause = 0;                        /* sweeps until the grid is sampled for a window (again) */
    uint32_t outside = 2u * JACOBI_SAMPLE;         /* sampled values outside the window, at the last failed sample */
    for (int s = 1; s <= job.sweeps; s++) {
        const double *u = owned ? owned : job.u0;
        double res = 0.0;
        int rc = 0;
        if (cells >= JACOBI_FIX_CELLS && !elow && ask-- == 0) {
            bool fp64;
            elow = jacobi_window(u, cells, &outside, &fp64, &rc);
            ask = pause;
            pause = min(2 * pause + 1, 15);
            if (rc)
                return 10;
            if (fp64 && gf_second_kernel((uint64_t)s, (uint64_t)owned))
                return 0;
        }
        double *un = jacobi_grid(job, s);
        if (!un)
            return 4;
        if (elow) {
            jacobi_red red, rest{0ull, 0, 0u};
            rc = gf_reduce<jacobi_red, GF_RED_MAX>(0, (int64_t)cut.warps * 32, GF_SCHED_STATIC, 1,
                                                   jacobi_fix_body{u, un, nn, elow, dn, dt, cut}, &red);
            if (!rc && red.out)
                rc = jacobi_rest(u, un, nn, cells, &rest);
            res = __longlong_as_double((long long)max(red.res, rest.res));
            const uint32_t hi = (uint32_t)max(red.hi, rest.hi), top = hi >> 20;
            if (red.out > cells / 64) {            /* the window does not suit: the FP64 pipe for a while */
                elow = 0u;
                ask = pause;
            } else {
                if (hi != 0u)                      /* 0: nothing but zeros was seen */
                    elow = top < 13u || top > GF_FIX_TOP ? 0u : top - 8u;
                ask = pause = 0;
            }
        } else {
            rc = cells >= JACOBI_FIX_CELLS ? jacobi_sweep_ahead(u, un, nn, dn, dsk, &res)
                                           : jacobi_sweep<0>(u, un, nn, dn, cells, &res);
        }
        if (rc)
            return 10;
        jacobi_swap(s, res, un, &owned);
    }
    return jacobi_write(job, owned);
}
