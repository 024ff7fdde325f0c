// kernels_smooth_f64_c.cu -- the double2 families of the line lengths in AFFT_SMOOTH_PLANS_C.
#include "kernel_tables.cuh"

namespace afft {

#define AFFT_X(N, ...) AFFT_SMOOTH_SET(double2, N, ##__VA_ARGS__)

const KernelSet *smooth_kernels_f64_c(int n)
{
    static const KernelSet table[] = {AFFT_SMOOTH_PLANS_C(AFFT_X)};
    return find_set(table, n);
}

}  // namespace afft
