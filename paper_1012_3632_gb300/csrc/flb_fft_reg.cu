// flb_fft_reg.cu -- one part of the lengths of flb_fft_reg.cuh, compiled once per
// part with FLB_REG_PART = 0, 1, ..: a process loads the parts whose lengths it
// uses.
#include <utility>

#ifndef FLB_REG_PART
#define FLB_REG_PART 0
#endif

#include "flb_fft_reg.cuh"

namespace flb {
namespace {

template <int L>
constexpr RegKernels kernels_of()
{
    return {L, kRegLines<L>, kRegThreads<L>, k_fft_rows<L>, k_fft_strided<L, false>, k_fft_strided<L, true>,
            k_swift_columns<L>};
}
constexpr int kCount = (kRegLengths - FLB_REG_PART + kRegParts - 1) / kRegParts;

template <class I>
struct Part;
template <int... I>
struct Part<std::integer_sequence<int, I...>> {
    static constexpr RegKernels table[] = {kernels_of<reg_length(FLB_REG_PART + I * kRegParts)>()...};
};

}  // namespace

#define FLB_REG_NAME2(K) reg_part_##K
#define FLB_REG_NAME(K) FLB_REG_NAME2(K)
const RegKernels* FLB_REG_NAME(FLB_REG_PART)() { return Part<std::make_integer_sequence<int, kCount>>::table; }

}  // namespace flb
