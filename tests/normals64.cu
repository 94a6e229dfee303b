// Test helper: the FP64 paths' Box-Muller (csrc/flb_normal64.cuh) on a list of
// word pairs, and the same by the CUDA math library.
#include "../paper_1012_3632_gb300/csrc/flb_device.cuh"

__global__ void k_normals(const uint2* w, int n, double2* out, double2* lib)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    flb::box_muller(w[i].x, w[i].y, out[i].x, out[i].y);
    const double u0 = ((double)w[i].x + 0.5) * 2.3283064365386963e-10, u1 = ((double)w[i].y + 0.5) * 2.3283064365386963e-10;
    const double r = sqrt(-2.0 * log(u0));
    double s, c;
    sincospi(2.0 * u1, &s, &c);
    lib[i] = make_double2(r * c, r * s);
}

extern "C" int normals64(const unsigned* words, int n, double* out, double* lib)
{
    uint2* d_w = nullptr;
    double2 *d_o = nullptr, *d_l = nullptr;
    cudaError_t e = cudaMalloc(&d_w, n * sizeof(uint2));
    if (e == cudaSuccess) e = cudaMalloc(&d_o, n * sizeof(double2));
    if (e == cudaSuccess) e = cudaMalloc(&d_l, n * sizeof(double2));
    if (e == cudaSuccess) e = cudaMemcpy(d_w, words, n * sizeof(uint2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_normals<<<(n + 127) / 128, 128>>>(d_w, n, d_o, d_l);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d_o, n * sizeof(double2), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(lib, d_l, n * sizeof(double2), cudaMemcpyDeviceToHost);
    cudaFree(d_w);
    cudaFree(d_o);
    cudaFree(d_l);
    return (int)e;
}
