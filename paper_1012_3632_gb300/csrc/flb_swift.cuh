// flb_swift.cuh -- the white noise under the modified equilibrium's coloured noise.
#pragma once

#include "flb_device.cuh"

namespace flb {

// z_e + i z_eps of a site: normals 0 and 5 of the D2Q9 collision draw (calls 0
// and 1 of tag 0): Box-Muller in FP64 for double2 and in FP32 for float2, as the
// collision kernels of those precisions draw them.
template <class T>
__device__ __forceinline__ T swift_white(const PhiloxKeys& key, uint32_t site, uint32_t step, uint32_t replica)
{
    using E = decltype(T::x);
    E a[2], b[2];
    normal_pair(key, site, step, 0, replica, a[0], a[1]);
    normal_pair(key, site, step, 2, replica, b[0], b[1]);
    return T{a[0], b[1]};
}

// FP32 noise field in three passes over it (flb_fft.cu), where both lengths have
// a register plan: the white noise into the x transform, both y transforms with
// the colouring between them, the x transform.  chol: (c11, c21, c22) per
// wavevector; out as swift_noise leaves it, work: X Y complex numbers.
bool swift_noise_lengths(int X, int Y);
cudaError_t swift_noise_fp32(const PhiloxKeys& key, uint32_t step, uint32_t replica, int X, int Y, const float* chol,
                             float2* work, float2* out, cudaStream_t s);

}  // namespace flb
