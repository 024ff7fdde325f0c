"""radix_sequence (csrc/afft_internal.h), compiled for the host: for every 2/3/5-smooth line length the
radices multiply to the length, and one line's passes fit a generic CTA for every length but the
three that have never fitted (3888, 4000 and 4050 points, which plans refuse)."""
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
    for (int n = 1; n <= kMaxLine; ++n) {
        int m = n;
        for (int p : {2, 3, 5}) while (m %% p == 0) m /= p;
        int r[kMaxPasses];
        const int k = radix_sequence(n, r);
        if (m != 1) {
            if (k != -1) { printf("%%d is not smooth\n", n); return 1; }
            continue;
        }
        long long prod = 1;
        int threads = 1;
        for (int i = 0; i < k; ++i) {
            prod *= r[i];
            const int t = (n / r[i] + bmax_for_radix(r[i]) - 1) / bmax_for_radix(r[i]);
            threads = t > threads ? t : threads;
        }
        if (k < 0 || k > kMaxPasses || prod != n) { printf("%%d: wrong product\n", n); return 1; }
        if (threads > kGenericThreads) printf("refused %%d\n", n);
    }
    return 0;
}
'''


def test_radix_sequences_of_every_smooth_length(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "radix.cu"
    src.write_text(PROGRAM % HEADER)
    exe = str(tmp_path / "radix")
    subprocess.run([nvcc, "-std=c++17", "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert r.stdout.split() == ["refused", "3888", "refused", "4000", "refused", "4050"]
