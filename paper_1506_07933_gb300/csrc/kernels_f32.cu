// kernels_f32.cu -- instantiates the stage kernels for float2: one specialised
// family per line length of AFFT_LINE_PLANS, the strided-only sets of
// AFFT_STRIDED_PLANS_F32, and the generic family.
#include "kernel_tables.cuh"

namespace afft {

#define AFFT_X(N, ...) AFFT_KERNEL_SET(float2, false, N, ##__VA_ARGS__)

const KernelSet *spec_kernels_f32(int n)
{
    static const KernelSet table[] = {AFFT_LINE_PLANS(AFFT_X)};
    return find_set(table, n);
}

#undef AFFT_X
#define AFFT_X(N, ...)                                                                               \
    afft::kernel_set<afft::Spec<afft::LinePlan<N, ##__VA_ARGS__>>, float2, false>(                    \
        N, afft::LinePlan<N, ##__VA_ARGS__>::npass, afft::RadicesOf<afft::LinePlan<N, ##__VA_ARGS__>>::value),

const KernelSet *strided_kernels_f32(int n)
{
    static const KernelSet table[] = {AFFT_STRIDED_PLANS_F32(AFFT_X)};
    return find_set(table, n);
}

const KernelSet *generic_kernels_f32()
{
    static const KernelSet g = kernel_set<Generic, float2>(0, 0, nullptr);
    return &g;
}

}  // namespace afft
