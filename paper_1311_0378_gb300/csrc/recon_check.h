// Bounds-checked build (-DRECON_CHECKS, librecon_checks.so): the stand-in for a
// memory checker. RK_CHECK(cond, where) is cond, and counts a failure and keeps the
// where-code of the first; the caller skips the access instead of making it. In
// other builds it is true, and the branch around the access is gone. Every source
// file with kernels has its own counters (no relocatable device code);
// RK_CHECK_READER(name) defines the function that reads and resets them, which
// recon_checks (recon_kernels.cu) adds up.
#pragma once
#include <cuda_runtime.h>

enum {
    CK_QUEUE_SLOT = 1, CK_WAVEFRONT_PIXEL = 2, CK_PUSHED_PIXEL = 3,
    // merging engine
    CK_LABEL = 4,      // place of a label
    CK_BASIN = 5,      // basin number
    CK_PASS = 6,       // place in the pass list, of a pass in the block, or in the list of joins
    CK_LIVE = 7,       // place in a list of live roots
    CK_SLOT = 8,       // node slot of the block
    CK_NODE = 9,       // node number, or block number behind one
    // distance transform
    CK_WORD = 10,      // place in the column masks
    CK_COLUMN = 11,    // place in the column distances
    CK_ROW = 12        // column of the row in shared memory
};

typedef cudaError_t (*check_reader)(unsigned *violations, unsigned *first, int reset);
cudaError_t rk_read_checks(unsigned *violations, unsigned *first, int reset);
cudaError_t rf_read_checks(unsigned *violations, unsigned *first, int reset);
cudaError_t dt_read_checks(unsigned *violations, unsigned *first, int reset);

#ifdef RECON_CHECKS
namespace {
__device__ unsigned g_check[2];   // failed checks, where-code of the first
__device__ __noinline__ bool check_fail(unsigned where)
{
    atomicAdd(&g_check[0], 1u);
    atomicCAS(&g_check[1], 0u, where);
    return false;
}
}  // namespace
#define RK_CHECK(cond, where) ((cond) ? true : check_fail(where))
#define RK_CHECK_READER(name)                                                                    \
    cudaError_t name(unsigned *violations, unsigned *first, int reset)                           \
    {                                                                                            \
        unsigned v[2];                                                                           \
        cudaError_t e = cudaMemcpyFromSymbol(v, g_check, sizeof(v));                             \
        if (e != cudaSuccess) return e;                                                          \
        *violations = v[0];                                                                      \
        *first = v[1];                                                                           \
        const unsigned z[2] = {0u, 0u};                                                          \
        return reset ? cudaMemcpyToSymbol(g_check, z, sizeof(z)) : cudaSuccess;                  \
    }
#else
#define RK_CHECK(cond, where) true
#define RK_CHECK_READER(name)
#endif
