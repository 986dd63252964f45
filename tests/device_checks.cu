// Device functions of the integrator, evaluated on host arrays for
// test_gpu_device_math.py (compiled by it with the flags of the kernels'
// own units).
#include <cstdint>

#include "bd_launch.h"
#include "bd_lj.cuh"

using namespace bdra;

namespace {

constexpr int kFields = 1 << 21;

// A generator output whose six 21-bit fields are f[0..5] (Fields21).
__device__ uint4 with_fields(const uint32_t (&f)[6])
{
    return make_uint4(f[0] << 11 | f[4] >> 10, f[1] << 11 | (f[4] & 0x3FFu), f[2] << 11 | f[5] >> 10, f[3] << 11 | (f[5] & 0x3FFu));
}

// Draw i has radius fields i and angle fields that run through every value
// with i (an odd factor permutes them), other ones in each of the three pairs.
__global__ void noise_kernel(StepParams p, unsigned long long* bad)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, mask = kFields - 1;
    if (i >= (uint32_t)kFields) return;
    uint32_t f[6];
    for (int k = 0; k < 3; ++k) {
        f[2 * k] = (i + 699051u * k) & mask;
        f[2 * k + 1] = (i * (1664525u + 4u * k) + 374761u * k) & mask;
    }
    const uint4 x = with_fields(f);
    unsigned long long n = 0;
    for (int k = 0; k < 6; ++k) n += Fields21::m(x, k) != f[k];
    double a[6], b[6];
    draw_half<double, false, 0>(x, 0u, p, a[0], a[1], a[2]);
    draw_half<double, false, 1>(x, 1u, p, a[3], a[4], a[5]);
    Normals<double, false>::draw(x, 0u, b[0], b[1], b[2]);
    Normals<double, false>::draw(x, 1u, b[3], b[4], b[5]);
    for (int k = 0; k < 6; ++k) n += __double_as_longlong(a[k]) != __double_as_longlong(b[k]);
    if (n) atomicAdd(bad, n);
}

__global__ void spring_kernel(int64_t n, const double* q, double H, double Hinvb, double smin, double* c, int32_t* floored)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int fl = 0;
    c[i] = spring_coef<double, false>(q[3 * i], q[3 * i + 1], q[3 * i + 2], H, Hinvb, smin, fl);
    floored[i] = fl;
}

__global__ void recip_kernel(int64_t n, const double* x, double* y)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = Rsqrt<double, false>::rcp(x[i]);
}

template <typename T> struct Dev {      // device copy of a host array
    T* p = nullptr;
    size_t bytes;
    Dev(const T* host, int64_t n) : bytes(sizeof(T) * (size_t)n)
    {
        if (cudaMalloc(&p, bytes) == cudaSuccess && host) cudaMemcpy(p, host, bytes, cudaMemcpyHostToDevice);
    }
    ~Dev() { cudaFree(p); }
};

int blocks(int64_t n) { return (int)((n + 255) / 256); }

}  // namespace

extern "C" {

// Values that differ between the integrator's float64 draw and Box-Muller by the library functions, over every 21-bit field.
int check_noise(unsigned long long* mismatches)
{
    const unsigned long long zero = 0;
    Dev<char> rad(nullptr, (int64_t)noise_rad_bytes()), ang(nullptr, (int64_t)noise_ang_bytes());
    Dev<unsigned long long> bad(&zero, 1);
    if (!rad.p || !ang.p || !bad.p) return 1;
    if (run_noise_tables(rad.p, ang.p, nullptr) != cudaSuccess) return 2;
    StepParams p = {};
    p.rad_tab = (const double*)rad.p;
    p.ang_tab = (const double2*)ang.p;
    noise_kernel<<<blocks(kFields), 256>>>(p, bad.p);
    return cudaMemcpy(mismatches, bad.p, sizeof(*mismatches), cudaMemcpyDeviceToHost) != cudaSuccess;
}

int check_spring(int64_t n, const double* q, double H, double Hinvb, double smin, double* c, int32_t* floored)
{
    Dev<double> dq(q, 3 * n), dc(nullptr, n);
    Dev<int32_t> df(nullptr, n);
    if (!dq.p || !dc.p || !df.p) return 1;
    spring_kernel<<<blocks(n), 256>>>(n, dq.p, H, Hinvb, smin, dc.p, df.p);
    if (cudaMemcpy(c, dc.p, dc.bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    return cudaMemcpy(floored, df.p, df.bytes, cudaMemcpyDeviceToHost) != cudaSuccess;
}

int check_recip(int64_t n, const double* x, double* y)
{
    Dev<double> dx(x, n), dy(nullptr, n);
    if (!dx.p || !dy.p) return 1;
    recip_kernel<<<blocks(n), 256>>>(n, dx.p, dy.p);
    return cudaMemcpy(y, dy.p, dy.bytes, cudaMemcpyDeviceToHost) != cudaSuccess;
}

}  // extern "C"
