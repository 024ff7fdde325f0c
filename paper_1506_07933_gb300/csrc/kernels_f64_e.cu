// kernels_f64_e.cu -- the double2 specialised families of the line lengths in
// AFFT_LINE_PLANS_F64_E (the complex128 instantiations are the slowest to compile,
// so they are split over five translation units), and the strided-only sets of
// AFFT_STRIDED_PLANS_F64.
#include "kernel_tables.cuh"

namespace afft {

#define AFFT_X(N, ...) AFFT_KERNEL_SET(double2, false, N, ##__VA_ARGS__)

const KernelSet *spec_kernels_f64_e(int n)
{
    static const KernelSet table[] = {AFFT_LINE_PLANS_F64_E(AFFT_X)};
    return find_set(table, n);
}

#undef AFFT_X
#define AFFT_X(N, ...)                                                                               \
    afft::kernel_set<afft::Spec<afft::LinePlan<N, ##__VA_ARGS__>>, double2, false>(                   \
        N, afft::LinePlan<N, ##__VA_ARGS__>::npass, afft::RadicesOf<afft::LinePlan<N, ##__VA_ARGS__>>::value),

const KernelSet *strided_kernels_f64(int n)
{
    static const KernelSet table[] = {AFFT_STRIDED_PLANS_F64(AFFT_X)};
    return find_set(table, n);
}

}  // namespace afft
