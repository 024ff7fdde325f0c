"""Generic line kernels (lengths above 1024, four-step halves): both radix families, both layouts."""
import numpy as np
import pytest
import torch

import oracle
from paper_1506_07933_gb300 import afft, synth

pytestmark = pytest.mark.gpu

# complex64 against 64 bits; FP64 lines of at most 14 levels stay within a few eps sqrt(log2 n)
TOL = {"f32": 2e-6, "f64": 4e-15}
CDT = {"f32": np.complex64, "f64": np.complex128}
RDT = {"f32": np.float32, "f64": np.float64}


def check(shape, kind, prec, seed, tol=TOL):
    make = synth.uniform_complex if kind == "c2c" else synth.uniform_real
    x = make(shape, seed).astype((CDT if kind == "c2c" else RDT)[prec])
    ref = oracle.c2c(x, -1, "fft") if kind == "c2c" else oracle.r2c(x)
    with afft.Plan(shape, kind, prec) as p:
        radix = p.describe()["radix"]
        X = p.forward(torch.from_numpy(x).cuda())
        y = p.backward(torch.from_numpy(ref.astype(CDT[prec])).cuda())
        torch.cuda.synchronize()
    assert oracle.rel_l2(X.cpu().numpy(), ref) <= tol[prec], (shape, kind, prec, "forward")
    assert oracle.rel_l2(y.cpu().numpy(), x) <= tol[prec], (shape, kind, prec, "backward")
    return radix


@pytest.mark.parametrize("n,strided,contiguous", [
    (1280, {"f32": "16x16x5", "f64": "16x16x5"}, {"f32": "16x16x5", "f64": "16x16x5"}),
    (1920, {"f32": "16x8x3x5", "f64": "16x12x10"}, {"f32": "16x8x3x5", "f64": "16x12x10"}),
    (2000, {"f32": "16x5x5x5", "f64": "16x5x5x5"}, {"f32": "16x5x5x5", "f64": "16x5x5x5"}),
    (2187, {"f32": "9x9x9x3", "f64": "3x3x3x3x3x3x3"}, {"f32": "9x9x9x3", "f64": "3x3x3x3x3x3x3"}),
    (3375, {"f32": "15x15x15", "f64": "15x15x15"}, {"f32": "15x15x15", "f64": "15x15x15"}),
    (3645, {"f32": "15x3x3x3x3x3", "f64": "15x3x3x3x3x3"}, {"f32": "15x3x3x3x3x3", "f64": "15x3x3x3x3x3"})])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_lengths_of_both_families(n, strided, contiguous, prec):
    assert check((n, 2, 9), "c2c", prec, n)[0] == strided[prec]
    assert check((2, n, 5), "c2c", prec, n + 1)[1] == strided[prec]
    assert check((2, 3, n), "c2c", prec, n + 2)[2] == contiguous[prec]
    assert check((2, 3, 2 * n), "r2c", prec, n + 3)[2] == contiguous[prec]


@pytest.mark.parametrize("n", [4320, 5400, 5625, 6561, 12000])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_four_step_lengths(n, prec):
    tol = {"f32": 2e-6, "f64": 1e-12}   # the first half may be a float-float length
    check((n, 2, 5), "c2c", prec, n, tol)
    check((2, 3, n), "c2c", prec, n + 1, tol)


@pytest.mark.parametrize("shape", [(2, 432, 24), (3, 5, 720), (240, 4, 10)])
def test_generic_split_precision_lengths(shape):
    """Multiples of 16 without a split sequence: the generic kernels with tensor-core radix-16 passes."""
    x = synth.uniform_complex(shape, 3).astype(np.complex64)
    ref = oracle.c2c(x, -1, "fft")
    with afft.Plan(shape, "c2c", "f32_split") as p:
        assert p.describe()["specialised"][max(range(3), key=lambda a: shape[a])] == 0
        X = p.forward(torch.from_numpy(x).cuda())
        y = p.backward(torch.from_numpy(ref.astype(np.complex64)).cuda())
        torch.cuda.synchronize()
    assert oracle.rel_l2(X.cpu().numpy(), ref) <= 2e-5
    assert oracle.rel_l2(y.cpu().numpy(), x) <= 2e-5


@pytest.mark.parametrize("shape", [(1080, 3, 10), (3, 1125, 8), (2, 3, 2 * 1920)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_no_alloc_c2r_with_generic_lengths(shape, prec):
    x = synth.uniform_real(shape, 5)
    X = torch.from_numpy(oracle.r2c(x).astype(CDT[prec])).cuda()
    y = torch.empty(shape, dtype=torch.float32 if prec == "f32" else torch.float64, device="cuda")
    afft.afft_c2r_noalloc(shape, afft.F32 if prec == "f32" else afft.F64, X.data_ptr(), y.data_ptr(),
                          torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert oracle.rel_l2(y.cpu().numpy(), x) <= TOL[prec]
