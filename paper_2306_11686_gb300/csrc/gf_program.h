/*
 * Program registry: GF_MAIN(name) registers, at load time of the object that
 * defines it, a cooperative launcher and an occupancy query for the program's
 * persistent kernel, and a launcher of its region kernel (the kernel split,
 * used when a context runs with split_regions).  Keeping the launch inside the defining translation unit
 * lets programs live in any shared object linked against the runtime.
 */
#ifndef GF_PROGRAM_H
#define GF_PROGRAM_H
#include <cuda_runtime.h>

typedef cudaError_t (*gf_launch_fn)(void **args, unsigned grid, unsigned block, void *stream);
typedef int (*gf_occ_fn)(unsigned block);
/* which kernels a launch of a program with a second kernel takes */
enum { GF_FIRST_ONLY = 0, GF_SECOND_ONLY = 1, GF_BOTH = 2 };
typedef int (*gf_pick_fn)(int argc, const char *const *argv);

#ifdef __cplusplus
extern "C"
#endif
    __attribute__((visibility("default"))) int
    gf_program_register(const char *name, gf_launch_fn launch, gf_occ_fn occ, gf_launch_fn region);

/* A second kernel for the program `name`, compiled for another number of resident
 * blocks; registered before or after the program itself.  pick(argc, argv) says which of the two a launch takes; with
 * GF_BOTH the second one is queued behind the first and goes on where the
 * first one's main called gf_second_kernel, or ends at once. */
#ifdef __cplusplus
extern "C"
#endif
    __attribute__((visibility("default"))) int
    gf_program_second(const char *name, gf_pick_fn pick, gf_launch_fn launch, gf_occ_fn occ, gf_launch_fn region);

#endif
