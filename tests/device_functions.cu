// Device functions of the library over their whole ranges, one check a call; built
// and run by test_gpu_device_functions.py.
#include <cstdio>
#include <cstring>

#include "hfs_fno_frag.cuh"
#include "hfs_phase.cuh"

using namespace hfs;

__device__ void atomic_max(double *p, double v)  // of values >= 0
{
    atomicMax(reinterpret_cast<unsigned long long *>(p), (unsigned long long)__double_as_longlong(v));
}

// apply_turns in FP64 against sincospi: turns over 2^-60 .. 2^40 (uniform in the
// exponent) of either sign
__global__ void turns_error(double *worst)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    const double turns = (i & 1 ? -1.0 : 1.0) * exp2(-60.0 + 100.0 * i / n);
    const cpx<double> v = apply_turns(cpx<double>{1.0, 0.0}, turns, 1.0);
    double s, c;
    sincospi(2.0 * (turns - rint(turns)), &s, &c);
    atomic_max(worst, fmax(fabs(v.x - c), fabs(v.y + s)));
}

// its modulus over all finite turns
__global__ void turns_modulus(double *worst)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    const double turns = (i & 1 ? -1.0 : 1.0) * exp2(-1000.0 + 2023.9 * i / n);
    const cpx<double> v = apply_turns(cpx<double>{0.8, -0.6}, turns, 1.0);
    const double e = fabs(v.x * v.x + v.y * v.y - 1.0);
    atomic_max(worst, e >= 0.0 ? e : 1e300);
}

// gelu4 against bf16(gelu_f) over all 2^32 values of z, in each of its four places:
// values that differ
__global__ void gelu_differences(double *count)
{
    const unsigned long long n = gridDim.x * (unsigned long long)blockDim.x;
    unsigned long long bad = 0;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < (1ull << 32); i += n) {
        const float z = __uint_as_float((unsigned)i), o = 0.5f;
        const unsigned ref = fno::pack2(fno::gelu_f(z), fno::gelu_f(o));
        const uint2 a = fno::gelu4(z, o, 1.0f, 2.0f), b = fno::gelu4(1.0f, 2.0f, z, o);
        const uint2 c = fno::gelu4(o, z, 1.0f, 2.0f), d = fno::gelu4(1.0f, 2.0f, o, z);
        const unsigned swapped = ref << 16 | ref >> 16;
        bad += a.x != ref || b.y != ref || c.x != swapped || d.y != swapped;
    }
    atomicAdd(count, (double)bad);
}

int main(int, char **argv)
{
    double *d = nullptr, h = 0.0;
    if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 1;
    if (!strcmp(argv[1], "turns_error")) turns_error<<<4096, 256>>>(d);
    else if (!strcmp(argv[1], "turns_modulus")) turns_modulus<<<4096, 256>>>(d);
    else if (!strcmp(argv[1], "gelu_differences")) gelu_differences<<<1520, 256>>>(d);
    else return 1;
    if (cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%.17g\n", h);
    return cudaFree(d) != cudaSuccess;
}
