"""Line lengths with prime factors 2, 3, 5 that are not in the main table (AFFT_SMOOTH_PLANS): every
length up to 1024 on every axis and in every kernel it can take, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1506_07933_gb300 import afft, synth

pytestmark = pytest.mark.gpu


def smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


MAIN = {2, 4, 8, 16, 24, 32, 48, 60, 64, 80, 96, 120, 128, 160, 192, 256, 384, 512, 1024}
LENGTHS = [n for n in range(2, 1025) if smooth(n) and n not in MAIN]
# five-smooth lengths of the generic kernels with radices 6, 9, 10, 12 and 15 among their passes
# (2430 ... 3750: lengths whose shortest sequences do not fit a CTA)
GENERIC = [1080, 1125, 1458, 1728, 3125, 2430, 2592, 2916, 3000, 3200, 3240, 3456, 3645, 3750]
# FP64 lines of these lengths compute in FP64: a length-n FFT of log2(n) <= 12 levels stays within a
# few eps sqrt(log2 n), far below the float-float kernels' 1e-14
TOL = {"f32": 2e-6, "f64": 4e-15}
CDT = {"f32": np.complex64, "f64": np.complex128}
RDT = {"f32": np.float32, "f64": np.float64}


def check(shape, kind, prec, seed):
    make = synth.uniform_complex if kind == "c2c" else synth.uniform_real
    x = make(shape, seed).astype((CDT if kind == "c2c" else RDT)[prec])
    ref = oracle.c2c(x, -1, "fft") if kind == "c2c" else oracle.r2c(x)
    with afft.Plan(shape, kind, prec) as p:
        X = p.forward(torch.from_numpy(x).cuda())
        y = p.backward(torch.from_numpy(ref.astype(CDT[prec])).cuda())
        torch.cuda.synchronize()
        assert p.device_status() == 0
    assert oracle.rel_l2(X.cpu().numpy(), ref) <= TOL[prec], (shape, kind, prec, "forward")
    assert oracle.rel_l2(y.cpu().numpy(), x) <= TOL[prec], (shape, kind, prec, "backward")


@pytest.mark.parametrize("n", LENGTHS + GENERIC)
def test_length_on_every_axis(n):
    for prec in ("f32", "f64"):
        check((n, 4, 10), "c2c", prec, n)          # N0: TMA tiles, the last one ragged
        check((2, n, 25), "c2c", prec, n + 1)      # N1: rows of odd width (row pairs, or no tensor map)
        check((3, 5, n), "c2c", prec, n + 2)       # N2: whole lines
        check((3, n, 36), "r2c", prec, n + 3)      # N1 of an r2c plan: 19 bins per row
        check((2, 5, 2 * n), "r2c", prec, n + 4)   # half-length lines of r2c and c2r


@pytest.mark.parametrize("kind,prec", [("r2c", "f32"), ("c2c", "f64")])
def test_chained_launches_in_a_captured_graph(kind, prec):
    """Stage kernels start before their predecessor ends: forward, backward and an overwrite of the
    input, replayed from a user's graph and back to back on the stream, give the same bits each time."""
    shape = (40, 36, 48)
    rng = np.random.default_rng(5)
    xs = []
    for _ in range(3):
        x = rng.uniform(-1, 1, shape)
        xs.append((x + 1j * rng.uniform(-1, 1, shape) if kind == "c2c" else x).astype((CDT if kind == "c2c" else RDT)[prec]))
    xs = [torch.from_numpy(x).cuda() for x in xs]
    with afft.Plan(shape, kind, prec) as p:
        want = []
        for x in xs:
            X = p.forward(x)
            torch.cuda.synchronize()
            y = p.backward(X)
            torch.cuda.synchronize()
            want.append((X, y))
        buf = torch.empty_like(xs[0])
        X = torch.empty(p.spectral_shape, dtype=p.spectral_dtype, device="cuda")
        y = torch.empty_like(buf)
        got = []
        for x in xs:                      # one stream, nothing waited for in between
            buf.copy_(x)
            p.backward(p.forward(buf, out=X), out=y)
            got.append((X.clone(), y.clone()))
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            y.zero_()
            p.backward(p.forward(buf, out=X), out=y)
            y2 = y + 0
        for x in xs:
            buf.copy_(x)
            g.replay()
            got.append((X.clone(), y2.clone()))
        torch.cuda.synchronize()
        for i, (a, b) in enumerate(got):
            assert torch.equal(a, want[i % 3][0]) and torch.equal(b, want[i % 3][1]), i
    assert oracle.rel_l2(want[0][1].cpu().numpy(), xs[0].cpu().numpy()) <= (2e-6 if prec == "f32" else 1e-12)


@pytest.mark.parametrize("n", [1] + sorted(MAIN | set(LENGTHS)))
def test_poisson_every_n0_length(n):
    """The fused N0 operator (forward, 1/|k|^2 and inverse in one middle pass) at every line length,
    with a ragged last tile, and rows of odd width (which take the separate multiply)."""
    for shape in ((n, 6, 12), (n, 5, 12)):
        for prec in ("f32", "f64"):
            f = synth.uniform_real(shape, n).astype(RDT[prec])
            with afft.Plan(shape, "r2c", prec) as p:
                u = p.poisson(torch.from_numpy(f).cuda())
                torch.cuda.synchronize()
                assert p.device_status() == 0
            err = oracle.rel_l2(u.cpu().numpy(), oracle.poisson(f.astype(np.float64)))
            assert err <= (2e-6 if prec == "f32" else 1e-12), (shape, prec, err)


def test_length_with_a_strided_and_a_contiguous_sequence():
    """160 points in complex64: strided stages 10 x 16, contiguous lines 16 x 10."""
    check((160, 4, 10), "c2c", "f32", 1)
    check((2, 160, 25), "c2c", "f32", 2)
    check((3, 160, 160), "c2c", "f32", 3)
    check((2, 5, 320), "r2c", "f32", 4)
    with afft.Plan((160, 160, 160), "c2c", "f32") as p:
        assert p.describe()["radix"] == ["10x16", "10x16", "16x10"]
