/*
 * Host-only test of a launch's device state: runtime.cu compiled against a
 * fake CUDA runtime whose device memory is host memory of exactly the sizes
 * asked for, and whose stream holds the reset kernel back until something
 * waits for the stream.
 *
 *   launch_fake_cuda <scenario>
 *
 * Scenarios (each prints "OK" and exits 0, or prints the failure and exits 1):
 *   reset    what the reset kernel is told to write lies inside the
 *            allocations, over configurations whose arrays are small or odd
 *   failed   a launch or a borrow that fails after the reset kernel was queued
 *            gives the instance back only when that kernel has run
 *   split    the state of a program whose regions are kernels of their own
 *            counts the threads of the region kernel as workers
 *   clear    the heap's metadata and the format cache are zero when the program
 *            starts, in contexts for one program and for several
 *   second   which kernels a launch of a program with two takes, on what grids
 */
#include <cuda_runtime.h>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace fake {
std::map<uint64_t, uint64_t> mem;                 /* allocations: address, bytes asked for */
struct Kernel {
    cudaStream_t stream;
    std::vector<char> args;
};
std::vector<Kernel> queued;                       /* reset kernels that have not run */
std::string trouble;
size_t arg_bytes = 0;
void run(const std::vector<char> &args);          /* the reset kernel on the host */

template <class T> cudaError_t alloc(T **p, size_t n)
{
    *p = (T *)calloc(1, n + 64);
    mem[(uint64_t)*p] = n;
    return cudaSuccess;
}
cudaError_t release(void *p)
{
    mem.erase((uint64_t)p);
    free(p);
    return cudaSuccess;
}
bool inside(uint64_t a, uint64_t n)
{
    auto it = mem.upper_bound(a);
    return n == 0 || (it != mem.begin() && (--it, a + n <= it->first + it->second));
}
template <class T> cudaError_t make(T *p)
{
    *p = (T)malloc(1);
    return cudaSuccess;
}
cudaError_t drop(void *p)
{
    free(p);
    return cudaSuccess;
}
cudaError_t drain(cudaStream_t s)
{
    for (size_t k = 0; k < queued.size();)
        if (queued[k].stream == s) {
            run(queued[k].args);
            queued.erase(queued.begin() + (long)k);
        } else {
            k++;
        }
    return cudaSuccess;
}
cudaError_t launch(void **args, cudaStream_t s)
{
    const char *a = (const char *)args[0];
    queued.push_back({s, std::vector<char>(a, a + arg_bytes)});
    return cudaSuccess;
}
int copies_fail = 0;                              /* the next asynchronous copies fail */
cudaError_t copy(void *d, const void *s, size_t n, cudaStream_t st)
{
    if (copies_fail) {
        copies_fail--;
        return cudaErrorUnknown;
    }
    drain(st);
    memcpy(d, s, n);
    return cudaSuccess;
}
template <class T> cudaError_t is(T *p, T v)
{
    *p = v;
    return cudaSuccess;
}
cudaError_t clear(void *d, size_t n)
{
    if (!inside((uint64_t)d, n))
        trouble += "a memset reaches past its allocation\n";
    else
        memset(d, 0, n);
    return cudaSuccess;
}
cudaError_t dev_pointer(cudaPointerAttributes *a)
{
    memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
} // namespace fake

#define cudaMalloc(p, n) fake::alloc(p, n)
#define cudaMallocAsync(p, n, s) fake::alloc(p, n)
#define cudaHostAlloc(p, n, f) fake::alloc(p, n)
#define cudaFree(p) fake::release(p)
#define cudaFreeAsync(p, s) fake::release(p)
#define cudaFreeHost(p) fake::release(p)
#define cudaHostGetDevicePointer(d, h, f) fake::is((void **)(d), (void *)(h))
#define cudaPointerGetAttributes(a, p) fake::dev_pointer(a)
#define cudaStreamCreateWithFlags(s, f) fake::make(s)
#define cudaEventCreateWithFlags(e, f) fake::make(e)
#define cudaStreamDestroy(s) fake::drop(s)
#define cudaEventDestroy(e) fake::drop(e)
#define cudaEventRecord(e, s) cudaSuccess
#define cudaEventQuery(e) cudaSuccess
#define cudaEventSynchronize(e) cudaSuccess
#define cudaStreamSynchronize(s) fake::drain(s)
#define cudaMemcpyAsync(d, s, n, k, st) fake::copy((void *)(d), (const void *)(s), n, st)
#define cudaLaunchKernel(f, g, b, args, shm, s) fake::launch(args, s)
#define cudaMemsetAsync(d, v, n, s) fake::clear(d, n)
#define cudaSetDevice(d) cudaSuccess
#define cudaGetDevice(d) fake::is(d, 0)
#define cudaDeviceGetAttribute(v, a, d) fake::is(v, 152)
#define cudaDeviceGetLimit(v, l) fake::is(v, (size_t)4096)
#define cudaDeviceSetLimit(l, v) cudaSuccess

#include "runtime.cu"

void fake::run(const std::vector<char> &args)
{
    ResetArgs a;
    memcpy((void *)&a, args.data(), sizeof a);
    auto span = [&](const char *what, const void *p, uint64_t n) {
        if (!inside((uint64_t)p, n))
            trouble += std::string(what) + " reaches past its allocation\n";
    };
    span("state", a.state, a.init_n * 8ull);
    span("initial state", a.init, a.init_n * 8ull);
    span("argv", a.argv_to, a.argv_n * 8ull);
    span("argv source", a.argv_from, a.argv_n * 8ull);
    span("extents", a.ext, 8);
    for (int z = 0; z < 5; z++)
        span(("array " + std::to_string(z)).c_str(), a.zero[z], a.zero_n[z] * 16ull);
    if (!trouble.empty())
        return;
    memcpy(a.state, a.init, a.init_n * 8ull);
    memcpy(a.argv_to, a.argv_from, a.argv_n * 8ull);
    a.ext[0] = a.ext0;
    for (int z = 0; z < 5; z++)
        memset(a.zero[z], 0, a.zero_n[z] * 16ull);
}

static cudaError_t prog_launch(void **, unsigned, unsigned, void *) { return cudaSuccess; }
static cudaError_t prog_refused(void **, unsigned, unsigned, void *) { return cudaErrorUnknown; }
static int prog_occ(unsigned) { return 2; }

static int prog()
{
    return gf_program_register("fake", prog_launch, prog_occ, prog_launch);
}

static gf_config config()
{
    gf_config c;
    gf_config_default(&c);
    c.heap_bytes = 1 << 20;
    c.ring_slots = 8;
    c.server_threads = 0;
    c.bulk_bytes = 0;
    return c;
}

static bool reset()
{
    const int p = prog();
    const char *argv[2] = {"fake", "x"};
    for (uint64_t heap : {0ull, 1ull, 256ull << 10, 1ull << 20, (3ull << 20) + 1})
        for (uint32_t pct : {0u, 50u, 100u})
            for (uint32_t fmt : {1u, 2u, 4096u})
                for (int argc : {0, 1, 2}) {
                    gf_config cf = config();
                    cf.heap_bytes = heap;
                    cf.heap_small_pct = pct;
                    cf.fmt_cache = fmt;
                    gf_ctx *c = nullptr;
                    gf_handle *h = nullptr;
                    int ec = 0;
                    if (gf_init(&cf, &c) || gf_launch(c, p, argc, argv, nullptr, 0, nullptr, 0, &h) || gf_wait(h, &ec, 0))
                        fake::trouble += "a launch failed\n";
                    gf_finalize(c);
                    if (!fake::trouble.empty()) {
                        printf("heap %llu pct %u fmt_cache %u argc %d\n", (unsigned long long)heap, pct, fmt, argc);
                        return false;
                    }
                }
    return true;
}

static bool failed()
{
    const int good = prog(), bad = gf_program_register("refused", prog_refused, prog_occ, prog_launch);
    const gf_config cf = config();
    gf_ctx *c = nullptr;
    gf_handle *h = nullptr;
    int ec = 0, idx = -1, other = 0;
    if (gf_init(&cf, &c))
        return false;
    if (gf_launch(c, bad, 0, nullptr, nullptr, 0, &other, 0, &h) != GF_ECUDA || h)
        fake::trouble += "the refused launch did not fail\n";
    if (!fake::queued.empty())
        fake::trouble += "a failed launch leaves its reset kernel behind\n";
    fake::drain((cudaStream_t)&other);
    if (!gf_inst_acquire(c, &other, 1, &idx))
        return false;
    fake::copies_fail = 1;
    if (gf_inst_finish(c, idx, &other) != GF_ECUDA)
        fake::trouble += "the failed copy is not reported\n";
    if (!fake::queued.empty())
        fake::trouble += "a failed copy leaves the reset kernel behind\n";
    gf_inst_release(c, idx);
    fake::drain((cudaStream_t)&other);
    /* and the instance serves the next program */
    if (gf_launch(c, good, 0, nullptr, nullptr, 0, nullptr, 0, &h) || gf_wait(h, &ec, 0))
        fake::trouble += "the next launch failed\n";
    gf_finalize(c);
    return true;
}

static bool split()
{
    const int p = prog();
    for (uint32_t grid : {0u, 1u, 5u, 304u})
        for (uint32_t mode : {0u, 1u}) {
            gf_config cf = config();
            cf.split_regions = mode;
            cf.server_threads = 1;
            gf_ctx *c = nullptr;
            gf_handle *h = nullptr;
            int ec = 0;
            if (gf_init(&cf, &c) || gf_launch(c, p, 0, nullptr, nullptr, 0, nullptr, grid, &h))
                return false;
            const uint32_t all = grid ? grid : 304u;                       /* two blocks on each of 152 SMs */
            const uint32_t want = mode ? 256u * (all == 304u ? 303u : all) : 256u * all - 32u;
            const uint32_t got = h->inst->h_init()->nworkers;
            if (got != want) {
                printf("grid %u split %u: %u workers, not %u\n", grid, mode, got, want);
                return false;
            }
            if (gf_wait(h, &ec, 0))
                return false;
            gf_finalize(c);
        }
    return true;
}

static bool clear()
{
    const int p = prog();
    for (uint32_t programs : {1u, 3u}) {
        gf_config cf = config();
        cf.max_programs = programs;
        cf.heap_bytes = 3 << 20;
        gf_ctx *c = nullptr;
        if (gf_init(&cf, &c))
            return false;
        for (int turn = 0; turn < 2; turn++) {
            gf_handle *h = nullptr;
            int ec = 0;
            for (Instance *in : c->inst)
                for (void *a : {in->d_meta, in->d_heads, in->d_cur, in->d_lsize, in->d_fmt})
                    memset(a, 0x5a, fake::mem[(uint64_t)a]);
            if (gf_launch(c, p, 0, nullptr, nullptr, 0, nullptr, 0, &h))
                return false;
            fake::drain(h->stream);
            const Instance *in = h->inst;
            const struct {
                const void *at;
                size_t n;
            } want[] = {{in->d_meta, in->nslabs * 16ull},
                        {in->d_heads, (size_t)GF_MAX_SM * GF_HEAP_NCLASS * GF_HEAP_LANES * 8},
                        {in->d_cur, (size_t)GF_MAX_SM * GF_HEAP_NCLASS * 4},
                        {in->d_lsize, in->npages * 4ull},
                        {in->d_fmt, cf.fmt_cache * 8ull}};
            for (const auto &w : want)
                for (size_t k = 0; k < w.n; k++)
                    if (((const char *)w.at)[k]) {
                        printf("programs %u: a byte is left\n", programs);
                        return false;
                    }
            if (gf_wait(h, &ec, 0))
                return false;
        }
        gf_finalize(c);
    }
    return true;
}

static std::string launched;
static cudaError_t first_launch(void **, unsigned grid, unsigned, void *)
{
    launched += "first " + std::to_string(grid) + " ";
    return cudaSuccess;
}
static cudaError_t second_launch(void **, unsigned grid, unsigned, void *)
{
    launched += "second " + std::to_string(grid) + " ";
    return cudaSuccess;
}
static int second_occ(unsigned) { return 4; }
static int by_argc(int argc, const char *const *)
{
    return argc == 0 ? GF_BOTH : argc == 1 ? GF_SECOND_ONLY : GF_FIRST_ONLY;
}

static bool second()
{
    gf_program_second("two", by_argc, second_launch, second_occ, prog_launch);
    const int p = gf_program_register("two", first_launch, prog_occ, prog_launch);
    const struct {
        int argc;
        uint32_t programs, grid, split;
        const char *want;              /* launches, then the state's second and second_follows */
    } cases[] = {
        {0, 1, 0, 0, "first 304 second 608 0 1"}, {1, 1, 0, 0, "second 608 1 0"},   {2, 1, 0, 0, "first 304 0 0"},
        {0, 4, 0, 0, "first 76 second 152 0 1"},  {1, 4, 0, 0, "second 152 1 0"},   {0, 1, 100, 0, "first 100 second 200 0 1"},
        {1, 1, 100, 0, "second 100 1 0"},         {0, 1, 400, 0, "second 400 1 0"}, {2, 1, 608, 0, "second 608 1 0"},
        {0, 1, 609, 0, "refused"},                {1, 1, 609, 0, "refused"},        {0, 1, 0, 1, "first 1 0 0"},
        {1, 1, 0, 1, "second 1 1 0"},
    };
    const char *argv[2] = {"two", "x"};
    for (const auto &t : cases) {
        gf_config cf = config();
        cf.max_programs = t.programs;
        cf.split_regions = t.split;
        cf.server_threads = 1;
        gf_ctx *c = nullptr;
        gf_handle *h = nullptr;
        int ec = 0;
        if (gf_init(&cf, &c))
            return false;
        launched.clear();
        const int rc = gf_launch(c, p, t.argc, argv, nullptr, 0, nullptr, t.grid, &h);
        std::string got = rc == GF_EINVAL ? "refused" : launched;
        if (rc == GF_OK) {
            got += std::to_string(h->inst->h_init()->second) + " " + std::to_string(h->inst->h_init()->second_follows);
            gf_wait(h, &ec, 0);
        }
        if (got != t.want) {
            printf("argc %d programs %u grid %u split %u: %s, not %s\n", t.argc, t.programs, t.grid, t.split, got.c_str(),
                   t.want);
            return false;
        }
        gf_finalize(c);
    }
    return true;
}

int main(int argc, char **argv)
{
    fake::arg_bytes = sizeof(ResetArgs);
    const std::string s = argc > 1 ? argv[1] : "";
    const bool ok = s == "reset" ? reset() : s == "failed" ? failed() : s == "split" ? split() : s == "clear" ? clear() : s == "second" && second();
    printf("%s%s\n", fake::trouble.c_str(), ok && fake::trouble.empty() ? "OK" : "FAILED");
    return ok && fake::trouble.empty() ? 0 : 1;
}
