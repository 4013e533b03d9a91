// Checks of the checked build (-DSUPPY_CHECKED), one set of words a translation
// unit: CHECKED(cond, tag, idx) records the first violation (kernel tag, index)
// and is false, so that the access behind it is skipped.  Always true, and
// gone, in the ordinary build.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace suppy {
namespace {

#ifdef SUPPY_CHECKED
__device__ int g_check[3];   // {tag, index low, index high}
__device__ __noinline__ bool check_fail(int tag, long long idx) {
    if (atomicCAS(&g_check[0], 0, tag) == 0) {
        g_check[1] = (int)(idx & 0xffffffffLL);
        g_check[2] = (int)(idx >> 32);
    }
    return false;
}
#define CHECKED(cond, tag, idx) ((cond) ? true : check_fail((tag), (long long)(idx)))
#define ALIGNED16(p) ((((uintptr_t)(p)) & 15u) == 0)
#else
#define CHECKED(cond, tag, idx) true
#define ALIGNED16(p) true
#endif

// This unit's words, which go back to zero.
inline cudaError_t take_check_words(int* out3) {
#ifdef SUPPY_CHECKED
    cudaError_t e = cudaMemcpyFromSymbol(out3, g_check, sizeof(int) * 3);
    if (e != cudaSuccess) return e;
    const int z[3] = {0, 0, 0};
    return cudaMemcpyToSymbol(g_check, z, sizeof(int) * 3);
#else
    out3[0] = out3[1] = out3[2] = 0;
    return cudaSuccess;
#endif
}

}  // namespace
}  // namespace suppy
