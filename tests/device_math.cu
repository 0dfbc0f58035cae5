// The device arithmetic of fp64_math.cuh and hydro_math.cuh beside CUDA's own operations, one
// element per thread, for tests/test_gpu_device_math.py.
#include "hydro_math.cuh"

using namespace amr;

// pairs (a, b): o[0..n) recip(b), divide(a, b), sqrt_quot(a, b), minmod64(a, b), ge0(a), gt0(a)
// in blocks of n; w the same by CUDA's operations (minmod as the median of 0, a, b)
__global__ void k_ops(int64_t n, const double *a, const double *b, double *o, double *w)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const double x = a[i], y = b[i];
        o[i] = recip(y);
        o[n + i] = divide(x, y);
        o[2 * n + i] = sqrt_quot(x, y);
        o[3 * n + i] = minmod64(x, y);
        o[4 * n + i] = ge0(x);
        o[5 * n + i] = gt0(x);
        w[i] = 1.0 / y;
        w[n + i] = x / y;
        w[2 * n + i] = sqrt(x / y);
        w[3 * n + i] = fmax(fmin(x, y), fmin(fmax(x, y), 0.0));
        w[4 * n + i] = x >= 0.0;
        w[5 * n + i] = x > 0.0;
    }
}

// floor_at(a, f) and a > f ? a : f
__global__ void k_floor(int64_t n, const double *a, const double *f, double *o, double *w)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        o[i] = floor_at(a[i], f[i]);
        w[i] = a[i] > f[i] ? a[i] : f[i];
    }
}

// the FP32 kernels' reading of a state value, and the same by d2f_bits; both as the FP32 kernels'
// arithmetic sees them (denormals flushed by a multiplication)
__global__ void k_read(int64_t n, const double *x, float *o, float *w)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        o[i] = __fmul_rn(d2f_ftz(x[i]), 1.0f);
        w[i] = d2f_bits(x[i]);
    }
}

// x + f by add_f32 and by CUDA's conversion and addition
__global__ void k_add(int64_t n, const double *x, const float *f, double *o, double *w)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        o[i] = add_f32(x[i], f[i]);
        w[i] = __dadd_rn(x[i], double(f[i]));
    }
}

// how often cfl_step rises from one positive normal signal speed to the next
__global__ void k_monotone(float cfl, float dx, unsigned long long *rises)
{
    const int64_t first = 0x00800000, last = 0x7F7FFFFF;
    unsigned long long bad = 0;
    for (int64_t i = first + blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < last; i += int64_t(gridDim.x) * blockDim.x) {
        const double a = cfl_step(__int_as_float(int(i)), cfl, dx), b = cfl_step(__int_as_float(int(i + 1)), cfl, dx);
        bad += !(a >= b);
    }
    atomicAdd(rises, bad);
}

extern "C" int dm_ops(int64_t n, const double *a, const double *b, double *o, double *w)
{
    k_ops<<<304, 256>>>(n, a, b, o, w);
    return int(cudaDeviceSynchronize());
}
extern "C" int dm_floor(int64_t n, const double *a, const double *f, double *o, double *w)
{
    k_floor<<<304, 256>>>(n, a, f, o, w);
    return int(cudaDeviceSynchronize());
}
extern "C" int dm_read(int64_t n, const double *x, float *o, float *w)
{
    k_read<<<304, 256>>>(n, x, o, w);
    return int(cudaDeviceSynchronize());
}
extern "C" int dm_add(int64_t n, const double *x, const float *f, double *o, double *w)
{
    k_add<<<304, 256>>>(n, x, f, o, w);
    return int(cudaDeviceSynchronize());
}
extern "C" int dm_monotone(float cfl, float dx, unsigned long long *rises)
{
    k_monotone<<<1216, 256>>>(cfl, dx, rises);
    return int(cudaDeviceSynchronize());
}
