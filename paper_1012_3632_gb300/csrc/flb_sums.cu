// flb_sums.cu -- sums of the rows that the reductions leave.  A translation unit of
// its own: the first use of a kernel loads all that was compiled with it, and a
// run that only wants its totals should not wait for the transforms (the first
// flb_conservation of a process took 14 ms beside them, 0.2 here).
#include <algorithm>

#include "flb_internal.h"
#include "flb_kernels.cuh"

namespace flb {

// ---------------------------------------------------------------------------
// Column sums (one block per column, fixed order: deterministic)
// ---------------------------------------------------------------------------
__global__ void k_sum_columns(const double* partials, int nrows, int ncol, double* __restrict__ out,
                              double add0)
{
    __shared__ double sh[256];
    const int c = blockIdx.x;
    partials += (long)blockIdx.y * nrows * ncol;
    out += (long)blockIdx.y * ncol;
    pdl_wait();
    double acc = 0.0;
    for (int r = threadIdx.x; r < nrows; r += blockDim.x) acc += partials[(long)r * ncol + c];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[c] = c == 0 ? sh[0] + add0 : sh[0];
}

cudaError_t sum_columns(const double* partials, int nrows, int ncol, double* out, cudaStream_t s, double add0, int k)
{
    return launch_chain(k_sum_columns, dim3(ncol, k), dim3(256), s, partials, nrows, ncol, out, add0);
}

__global__ void __launch_bounds__(128) k_sum_lattices(const __grid_constant__ ModeSums a, int ncol,
                                                      double* __restrict__ out)
{
    __shared__ double sh[4];
    pdl_wait();
    const int c = blockIdx.x, r = blockIdx.y, end = a.lat[r + 1].first;
    double acc = 0.0;
    for (int k = a.lat[r].first + threadIdx.x; k < end; k += 128) acc += a.rows[(long)k * ncol + c];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) out[r * ncol + c] = (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

cudaError_t sum_lattices(const ModeSums& a, int ncol, double* out, cudaStream_t s)
{
    return launch_chain(k_sum_lattices, dim3(ncol, a.n), dim3(128), s, a, ncol, out);
}

// A load of what other blocks of this launch wrote (not from L1).
__device__ __forceinline__ double ld_relaxed(const double* p)
{
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

// Step blockIdx.y: its rows are split over gridDim.x blocks; the block that
// comes last adds their partial sums in block order (deterministic).
__global__ void __launch_bounds__(256) k_sum_steps(const float4* rows, int nrows, int per,
                                                   double* part, unsigned* ticks,
                                                   double* __restrict__ out, double add0)
{
    __shared__ double red[8][4];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, step = blockIdx.y, nb = gridDim.x;
    const float4* r = rows + (long)step * nrows;
    const int end = min(nrows, ((int)blockIdx.x + 1) * per);
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int k = blockIdx.x * per + threadIdx.x; k < end; k += 256) {
        const float4 f = r[k];
        v[0] += (double)f.x;
        v[1] += (double)f.y;
        v[2] += (double)f.z;
        v[3] += (double)f.w;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
    if (lane == 0)
        for (int c = 0; c < 4; ++c) red[warp][c] = v[c];
    __syncthreads();
    if (warp != 0) return;
    double acc = 0.0;
    if (lane < 4)
        for (int w = 0; w < 8; ++w) acc += red[w][lane];
    if (nb > 1) {
        double* p = part + 4 * (long)step * nb;
        if (lane < 4) p[4 * blockIdx.x + lane] = acc;
        __syncwarp();
        unsigned old = 0;
        if (lane == 0)
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(ticks + step) : "memory");
        if (__shfl_sync(0xffffffffu, old, 0) != (unsigned)nb - 1) return;
        __syncwarp();  // orders what lane 0 acquired before the loads of the others, a shuffle does not
        if (lane == 0) ticks[step] = 0u;
        acc = 0.0;
        for (int k = lane >> 2; k < nb; k += 8) acc += ld_relaxed(p + 4 * k + (lane & 3));
        for (int o = 16; o > 2; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    }
    if (lane < 4) out[4 * step + lane] = lane == 0 ? acc + add0 : acc;
}

cudaError_t sum_steps(const float4* rows, int nrows, int k, double* part, unsigned* ticks, double* out, double add0,
                      cudaStream_t s)
{
    // 2048 rows or more per block: 8 loads in flight per thread
    const int nb = std::min(kSumBlocksMax, (nrows + 2047) / 2048), per = (nrows + nb - 1) / nb;
    return launch_chain(k_sum_steps, dim3(nb, k), dim3(256), s, rows, nrows, per, part, ticks, out, add0);
}

}  // namespace flb
