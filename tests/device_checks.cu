// Device functions of the integrator, evaluated on host arrays for
// test_gpu_device_math.py (compiled by it with the flags of the kernels'
// own units).
#include <cstdint>

#include "bd_lj.cuh"

using namespace bdra;

namespace {

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
