// kernels_smooth_f32_e.cu -- the float2 families of the line lengths in AFFT_SMOOTH_PLANS_F32.
#include "kernel_tables.cuh"

namespace afft {

#define AFFT_X(N, ...) AFFT_SMOOTH_SET(float2, N, ##__VA_ARGS__)

const KernelSet *smooth_kernels_f32_e(int n)
{
    static const KernelSet table[] = {AFFT_SMOOTH_PLANS_F32(AFFT_X)};
    return find_set(table, n);
}

}  // namespace afft
