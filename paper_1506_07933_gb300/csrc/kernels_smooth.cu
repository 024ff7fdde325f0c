// kernels_smooth.cu -- lookup of the smooth-length families (AFFT_SMOOTH_PLANS; five translation
// units per precision, so that they compile in parallel).
#include "afft_internal.h"

namespace afft {

const KernelSet *smooth_kernels_f32_a(int n);
const KernelSet *smooth_kernels_f32_b(int n);
const KernelSet *smooth_kernels_f32_c(int n);
const KernelSet *smooth_kernels_f32_d(int n);
const KernelSet *smooth_kernels_f32_e(int n);
const KernelSet *smooth_kernels_f64_a(int n);
const KernelSet *smooth_kernels_f64_b(int n);
const KernelSet *smooth_kernels_f64_c(int n);
const KernelSet *smooth_kernels_f64_d(int n);
const KernelSet *smooth_kernels_f64_e(int n);

const KernelSet *smooth_kernels_f32(int n)
{
    for (auto *f : {smooth_kernels_f32_a, smooth_kernels_f32_b, smooth_kernels_f32_c, smooth_kernels_f32_d,
                    smooth_kernels_f32_e})
        if (const KernelSet *k = f(n)) return k;
    return nullptr;
}

const KernelSet *smooth_kernels_f64(int n)
{
    for (auto *f : {smooth_kernels_f64_a, smooth_kernels_f64_b, smooth_kernels_f64_c, smooth_kernels_f64_d,
                    smooth_kernels_f64_e})
        if (const KernelSet *k = f(n)) return k;
    return nullptr;
}

}  // namespace afft
