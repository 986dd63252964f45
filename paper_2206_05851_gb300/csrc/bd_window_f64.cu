// Instantiations of the parent kernel and the persistent replica kernel for
// double state (bd_window.cuh, bd_window2.cuh, bd_persist.cuh). Compiled with
// -fmad=false.
#include "bd_persist.cuh"
#include "bd_launch.h"
#include "bd_variants.h"

namespace bdra {

namespace {
template <int L> const void* parent_fn(bool lj, bool block)
{
    if (block) return (const void*)parent_block_kernel<double, L, false>;
    if constexpr (L == 1) return nullptr;        // a tile of the block kernel only
    else return lj ? (const void*)parent_kernel<double, L, false, true> : (const void*)parent_kernel<double, L, false, false>;
}
}  // namespace

#define BD_PARENT_TILES(X) X(1) X(2) X(4) X(7) X(10) X(13) X(16)

const void* parent_func_f64(int L, bool lj, bool block)
{
    switch (L) {
#define X(l) case l: return parent_fn<l>(lj, block);
        BD_PARENT_TILES(X)
#undef X
    default: return nullptr;
    }
}

// Dynamic shared memory of a block-kernel CTA, allowed here for the current device.
cudaError_t parent_block_smem_f64(int L, size_t* bytes)
{
    *bytes = 0;
    switch (L) {
#define X(l) case l: *bytes = ParentBlock<double, l>::bytes; break;
        BD_PARENT_TILES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
    return cudaFuncSetAttribute(parent_func_f64(L, false, true), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*bytes);
}

const void* persist_plain_f64(int v)
{
    switch (v) {
#define X(x) case x: return (const void*)replica_persist_kernel<double, false, x, false>;
        BD_VARIANTS_F64(X)
#undef X
    default: return nullptr;
    }
}

const void* persist_func_f64(int v, bool conf)
{
    return conf ? persist_conf_f64(v) : persist_plain_f64(v);
}

namespace {
// NoiseTab's entries, by the expressions of bm_pair.
__global__ void noise_tables_kernel(double* rad, double2* ang)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const double u = ((double)m + 0.5) * 4.76837158203125e-7;      // (m + 1/2) 2^-21
    if (m < NoiseTab::kRad) rad[m] = sqrt(-2.0 * log(u));
    if (m < NoiseTab::kAng) {
        double s, c;
        sincospi(2.0 * u, &s, &c);
        ang[m] = make_double2(c, s);
    }
}
}  // namespace

size_t noise_rad_bytes() { return sizeof(double) * NoiseTab::kRad; }
size_t noise_ang_bytes() { return sizeof(double2) * NoiseTab::kAng; }

cudaError_t run_noise_tables(void* rad, void* ang, cudaStream_t st)
{
    noise_tables_kernel<<<NoiseTab::kRad / 256, 256, 0, st>>>((double*)rad, (double2*)ang);
    return cudaGetLastError();
}

int persist_threads_f64() { return Persist<double>::threads; }

size_t persist_smem_f64(int v)
{
    switch (v) {
#define X(x) case x: return PersistSmem<double, false, x>::bytes;
        BD_VARIANTS_F64(X)
#undef X
    default: return 0;
    }
}

// Occupancy with the variant's dynamic shared memory, which is also allowed
// here (above the default 48 KiB) for the current device.
cudaError_t persist_blocks_per_sm_f64(int v, bool conf, int* n)
{
    const void* f = persist_func_f64(v, conf);
    if (!f) return cudaErrorInvalidValue;
    const size_t smem = persist_smem_f64(v);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, Persist<double>::threads, smem);
}

}  // namespace bdra
