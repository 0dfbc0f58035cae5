// csrc/launch.cuh against a fake of the CUDA runtime calls it makes: each line of output is a
// scenario, the status it returned, the launches made and the attribute calls made.
#include "launch.cuh"
#include <cstdio>

static int launches, attribute_calls;
static cudaError_t pending = cudaSuccess;      // what cudaGetLastError returns next
static cudaError_t next_launch = cudaSuccess;  // what the next launch returns (once)

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, enum cudaFuncAttribute, int) { ++attribute_calls; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = pending;
    pending = cudaSuccess;
    return e;
}
cudaError_t cudaLaunchKernel(const void *, dim3 g, dim3 b, void **args, size_t smem, cudaStream_t)
{
    if (g.x != 304 || b.x != 64 || smem != 100000 || *static_cast<int *>(args[0]) != 7) return cudaErrorUnknown;
    const cudaError_t e = next_launch;
    next_launch = cudaSuccess;
    if (e == cudaSuccess) ++launches;
    else pending = e;
    return e;
}
}

static void kern(int) {}

static void scenario(const char *name, cudaError_t launch, cudaError_t left_behind)
{
    next_launch = launch;
    pending = left_behind;
    launches = attribute_calls = 0;
    int arg = 7;
    const amr_status r = amr::launch_kernel(kern, 64, 100000, true, nullptr, arg,
                                            [](int64_t resident, int &) { return unsigned(resident); });
    std::printf("%s %d %d %d\n", name, int(r), launches, attribute_calls);
}

int main()
{
    scenario("first", cudaSuccess, cudaSuccess);
    scenario("cached", cudaSuccess, cudaSuccess);
    scenario("left_behind", cudaSuccess, cudaErrorInvalidValue);
    scenario("attributes_lost", cudaErrorInvalidValue, cudaSuccess);
    scenario("refused", cudaErrorInvalidConfiguration, cudaSuccess);
    scenario("after", cudaSuccess, cudaSuccess);
}
