// kernels_smooth_f64_e.cu -- the double2 families of the line lengths in AFFT_SMOOTH_PLANS_F64.
#include "kernel_tables.cuh"

namespace afft {

#define AFFT_X(N, ...) AFFT_SMOOTH_SET(double2, N, ##__VA_ARGS__)

const KernelSet *smooth_kernels_f64_e(int n)
{
    static const KernelSet table[] = {AFFT_SMOOTH_PLANS_F64(AFFT_X)};
    return find_set(table, n);
}

}  // namespace afft
