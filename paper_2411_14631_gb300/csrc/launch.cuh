// Launch of a kernel that needs dynamic shared memory and a grid of resident CTAs.  Host code.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime_api.h>
#include "../../include/amrhydro.h"

#define AMR_CUDA_TRY(expr)                                  \
    do {                                                    \
        cudaError_t e_ = (expr);                            \
        if (e_ != cudaSuccess) return AMR_ECUDA;            \
    } while (0)

namespace amr {

// How many of a kernel's CTAs with `smem` bytes are resident on the GPU at once, and its attributes
// set.  Both are properties of (kernel, device) and are looked up once per host thread: the three
// calls take some 20 us of host time, more than a small level's kernel.  After cudaDeviceReset the
// attributes are gone and the launch call itself returns cudaErrorInvalidValue: launch_kernel then
// sets them again and repeats it.
struct LaunchCache {
    struct Entry {
        const void *kern;
        int dev, resident;
    };
    Entry e[64];
    int n = 0;
};
inline LaunchCache &launch_cache()
{
    thread_local LaunchCache c;
    return c;
}
inline amr_status launch_setup(const void *kern, int threads, size_t smem, bool all_smem, int *resident)
{
    LaunchCache &c = launch_cache();
    int dev = 0, nsm = 0, per_sm = 0;
    AMR_CUDA_TRY(cudaGetDevice(&dev));
    for (int i = 0; i < c.n; ++i)
        if (c.e[i].kern == kern && c.e[i].dev == dev) {
            *resident = c.e[i].resident;
            return AMR_OK;
        }
    AMR_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    if (all_smem) AMR_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    AMR_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    *resident = per_sm * nsm;
    if (c.n < 64) c.e[c.n++] = {kern, dev, *resident};
    return AMR_OK;
}
// kern<<<grid(resident), threads, smem>>>(arg), grid computed from the resident CTAs.  The launch
// call's own error tells whether the kernel was launched; an error an earlier call left behind
// (cudaGetLastError) must not make it run twice, and is reported as AMR_ECUDA as everywhere.
template <typename A, typename G>
inline amr_status launch_kernel(void (*kern)(A), int threads, size_t smem, bool all_smem, cudaStream_t st, A &arg,
                                G grid)
{
    const void *fn = reinterpret_cast<const void *>(kern);
    for (int attempt = 0;; ++attempt) {
        int resident = 0;
        const amr_status r = launch_setup(fn, threads, smem, all_smem, &resident);
        if (r != AMR_OK) return r;
        const dim3 g(unsigned(grid(int64_t(resident), arg))), b{unsigned(threads)};
        void *args[] = {&arg};
        const cudaError_t e = cudaLaunchKernel(fn, g, b, args, smem, st);
        if (e == cudaSuccess) return cudaGetLastError() == cudaSuccess ? AMR_OK : AMR_ECUDA;
        (void)cudaGetLastError();
        if (e != cudaErrorInvalidValue || attempt) return AMR_ECUDA;
        launch_cache().n = 0;
    }
}

}  // namespace amr
