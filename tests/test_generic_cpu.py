"""mixed_pays (csrc/afft_internal.h), compiled for the host: which generic lines run radices 6 to 15."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1506_07933_gb300", "csrc", "afft_internal.h")

PROGRAM = r'''
#include <cstdio>
#include "%s"
using namespace afft;
int main()
{
    for (int n = 1025; n <= kMaxLine; ++n) {
        int m = n;
        for (int p : {2, 3, 5}) while (m %% p == 0) m /= p;
        if (m != 1) continue;
        for (int elem : {8, 16})
            for (int contiguous : {0, 1}) {
                int r[kMaxPasses];
                const bool mixed = mixed_pays(n, elem, contiguous);
                const int k = mixed ? radix_sequence(n, r) : basic_sequence(n, r);
                long long prod = 1;
                for (int i = 0; i < k; ++i) prod *= r[i];
                printf("%%d %%d %%d %%d %%d %%d\n", n, elem, contiguous, (int)mixed, prod == n && k <= kMaxPasses,
                       line_threads(r, k, n, 1) <= kGenericThreads);
            }
    }
    for (int n : {50, 60, 64, 72, 75, 80, 100})   // four-step halves
        for (int elem : {8, 16})
            printf("%%d %%d 2 %%d 1 1\n", n, elem, (int)mixed_pays(n, elem, false, 255));
    return 0;
}
'''


@pytest.fixture(scope="module")
def choices(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("generic")
    src, exe = d / "generic.cu", str(d / "generic")
    src.write_text(PROGRAM % HEADER)
    subprocess.run([nvcc, "-std=c++17", "-o", exe, str(src)], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return {tuple(map(int, l.split()[:3])): tuple(map(int, l.split()[3:])) for l in out.splitlines()}


def test_every_choice_is_a_sequence_that_fits(choices):
    assert len(choices) == 4 * 50 + 14
    for (n, elem, contiguous), (mixed, product, fits) in choices.items():
        assert product, n
        assert fits == (n not in (3888, 4000, 4050)), n


@pytest.mark.parametrize("n,elem,contiguous,mixed", [
    # the same passes, or as many: the mixed kernels only cost
    (3125, 8, 0, 0), (3125, 8, 1, 0), (3200, 16, 1, 0), (2000, 8, 0, 0), (2000, 8, 1, 0), (2000, 16, 0, 0),
    # fewer passes, but too few points in flight
    (1920, 8, 0, 0), (1920, 8, 1, 0), (1800, 8, 0, 0), (1600, 8, 0, 0), (1280, 8, 1, 0),
    # two radix-9 passes in complex128
    (1215, 16, 1, 0), (1458, 16, 0, 0),
    # the mixed kernels are faster
    (1080, 8, 0, 1), (1440, 8, 0, 1), (1800, 8, 1, 1), (2700, 8, 0, 1), (2700, 8, 1, 1), (2592, 16, 0, 1),
    (3375, 16, 1, 1),
    # four-step halves
    (72, 8, 2, 1), (75, 8, 2, 1), (75, 16, 2, 0), (50, 8, 2, 0), (60, 8, 2, 0), (64, 8, 2, 0), (100, 8, 2, 0)])
def test_choice(choices, n, elem, contiguous, mixed):
    assert choices[n, elem, contiguous][0] == mixed
