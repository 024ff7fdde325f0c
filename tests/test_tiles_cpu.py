"""Which strided tiles define their values on idle threads (PipeShape::define_singles, csrc/fft_pipe.cuh)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1506_07933_gb300", "csrc")

PROGRAM = r'''
#include "fft_pipe.cuh"
using namespace afft;
template <class P, class V> constexpr bool single = PipeShape<P, V>::define_singles;
template <class P> constexpr bool rows = RpShape<P>::define_singles;
// complex64: idle threads in a radix-16 pass, or full ones in 128-byte rows: measured slower when defined
static_assert(!single<LinePlan<48, 16, 3>, float2> && !single<LinePlan<80, 16, 5>, float2>, "");
static_assert(!single<LinePlan<384, 16, 8, 3>, float2> && !single<LinePlan<256, 16, 16>, float2>, "");
static_assert(!single<LinePlan<120, 8, 15>, float2> && !rows<LinePlan<256, 16, 16>>, "");
// 64-byte rows, row pairs, smooth lengths, complex128: measured faster
static_assert(single<LinePlan<1024, 16, 8, 8>, float2> && rows<LinePlan<128, 16, 8>> && rows<LinePlan<48, 16, 3>>, "");
static_assert(single<SmoothPlan<144, 16, 9>, float2> && single<LinePlan<48, 16, 3>, double2>, "");
int main() { return 0; }
'''


def test_tiles_that_define_their_values(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "tiles.cu"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), "-c", str(src), "-o", str(tmp_path / "tiles.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_lines_of_160_points():
    """Contiguous complex64 lines of 160 points start with radix 16 (10 first measured 142 us where 16 first
    takes 99), strided ones with radix 10."""
    text = open(os.path.join(CSRC, "fft_stage.cuh")).read()
    lines = text[text.index("#define AFFT_LINE_PLANS(X)"):]
    lines = lines[:lines.index("#define", 1)]
    assert "X(160, 16, 10)" in lines
    assert "#define AFFT_STRIDED_PLANS_F32(X) X(160, 10, 16)" in text
