// kernels_mixed.cu -- the generic families with radices 6, 9, 10, 12 and 15 (GenericMixed).
#include "fft_pipe.cuh"

namespace afft {

const KernelSet *mixed_kernels_f32()
{
    static const KernelSet g = kernel_set<GenericMixed, float2>(0, 0, nullptr);
    return &g;
}

const KernelSet *mixed_kernels_f64()
{
    static const KernelSet g = kernel_set<GenericMixed, double2>(0, 0, nullptr);
    return &g;
}

}  // namespace afft
