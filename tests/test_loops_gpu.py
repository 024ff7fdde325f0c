"""Every line length up to 1024 with more tiles than two rounds of resident CTAs, the last tile ragged: the second
load buffer, its barrier phases, reloads after an early release and the fused Poisson loop, which arrays of
a few tiles never reach, and contiguous CTAs of the ordinary size (more than 304 of them).  Against torch.fft
in 64 bits."""
import pytest
import torch

from paper_1506_07933_gb300 import afft

pytestmark = pytest.mark.gpu


def smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


LENGTHS = [n for n in range(2, 1025) if smooth(n)]
# complex64 a few eps sqrt(log2 n); complex128 lines in FP64 (the smooth lengths) or float-float
TOL = {"f32": 2e-6, "f64": 1e-12}
CDT = {"f32": torch.complex64, "f64": torch.complex128}


def rel(a, ref):
    return (torch.linalg.vector_norm(a.to(ref.dtype) - ref) / torch.linalg.vector_norm(ref)).item()


def field(plan, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty(plan.spatial_shape, dtype=plan.spatial_dtype, device="cuda")
    (torch.view_as_real(x) if x.is_complex() else x).uniform_(-1, 1, generator=g)
    return x


def resident(n, prec):
    """CTAs of the persistent kernel over lines of n points (0: the length has none)."""
    with afft.Plan((n, 1, 64), "c2c", prec, axes=1) as p:
        return p.describe()["pipe_ctas"][0]


def persistent(p, a):
    """The plan with axis a on its persistent kernel, where it has one but defaults to the plain one."""
    if not p.describe()["pipelined"][a]:
        cfg = p.tuning
        cfg[1 + a] = 1
        try:
            p.set_tuning(cfg)
        except afft.AfftError:
            pass
    return p


def check(p, dims, prec, seed):
    x = field(p, seed)
    wide = x.to(torch.complex128)
    ref = torch.fft.fftn(wide, dim=dims)
    X = p.forward(x)
    y = p.backward(ref.to(CDT[prec]).contiguous())
    torch.cuda.synchronize()
    assert p.device_status() == 0
    assert rel(X, ref) <= TOL[prec] and rel(y, wide) <= TOL[prec]


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_strided_tiles(n, prec):
    slots = max(152, resident(n, prec))
    per = 16 if prec == "f32" else 8
    # one slab of 2 slots tiles and a ragged one (even rows: TMA tiles; odd rows of odd n: plain kernels)
    for extra in (2, 3):
        with afft.Plan((n, 1, 2 * slots * per + extra), "c2c", prec, axes=1) as p:
            check(persistent(p, 0), (0,), prec, n)
    # slabs of rows of 25 columns: two row-pair tiles each where n is even
    with afft.Plan((2 * slots + 1, n, 25), "c2c", prec, axes=2) as p:
        check(persistent(p, 1), (1,), prec, n + 1)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_poisson_tiles(n, prec):
    slots = max(152, resident(n, prec))
    # 600 bins a slab: 37 tiles of 16 columns and one of eight
    tiles = 38 if prec == "f32" else 75
    batch = 2 * slots // tiles + 1
    with afft.Plan((n, 60, 18), "r2c", prec, batch=batch) as p:
        persistent(p, 0)
        f = field(p, n)
        u = p.poisson(f)
        torch.cuda.synchronize()
        assert p.device_status() == 0
    k = [torch.fft.fftfreq(m, 1.0 / m, dtype=torch.float64, device="cuda") for m in (n, 60)]
    k.append(torch.arange(10, dtype=torch.float64, device="cuda"))
    kk = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2] ** 2
    kk[0, 0, 0] = float("inf")
    dim = (-3, -2, -1)
    ref = torch.fft.irfftn(torch.fft.rfftn(f.double(), dim=dim) / kk, s=(n, 60, 18), dim=dim)
    assert rel(u, ref) <= TOL[prec]


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_contiguous_lines(n, prec):
    lines = 310 * (4096 if prec == "f32" else 2048) // n + 1
    with afft.Plan((lines, 1, n), "c2c", prec, axes=4) as p:
        check(p, (2,), prec, n)
    with afft.Plan((lines, 1, 2 * n), "r2c", prec, axes=4) as p:
        x = field(p, n)
        ref = torch.fft.rfft(x.double(), dim=2)
        X = p.forward(x)
        y = p.backward(ref.to(CDT[prec]).contiguous())
        torch.cuda.synchronize()
        assert p.device_status() == 0
        assert rel(X, ref) <= TOL[prec] and rel(y, x.double()) <= TOL[prec]


def test_the_kernels_these_shapes_run():
    """The persistent kernels are reached, the fused Poisson stage's through tuning where plans default to the
    plain ones; lengths without them (odd boxes of 64-byte rows, odd n in odd rows) run the plain kernel."""
    def kernels(shape, prec, axes, tuned=False):
        with afft.Plan(shape, "c2c", prec, axes=axes) as p:
            return (persistent(p, 0) if tuned else p).describe()["stage_kernels_forward"]
    assert kernels((243, 1, 4000), "f32", 1)[2] == "k_strided_pipe"
    assert kernels((9, 243, 25), "f32", 2)[1] == "k_strided"
    assert kernels((9, 250, 25), "f32", 2)[1] == "k_strided_pipe_rp"
    for n in (625, 675, 729):
        assert kernels((n, 1, 4000), "f32", 1)[2] == "k_strided"
    assert kernels((45, 1, 4000), "f64", 1)[2] == "k_strided"
    assert kernels((45, 1, 4000), "f64", 1, tuned=True)[2] == "k_strided_pipe"


@pytest.mark.parametrize("n", [45, 250, 243, 360, 625, 729])
def test_bases_of_8_bytes(n, prec="f32"):
    """Complex64 arrays that start 8 bytes past a 16-byte boundary, which no tensor map covers."""
    for shape, axes, dim in (((n, 1, 4100), 1, 0), ((40, n, 25), 2, 1), ((40, n, 26), 2, 1), ((100, 1, n), 4, 2)):
        with afft.Plan(shape, "c2c", prec, axes=axes) as p:
            size = shape[0] * shape[1] * shape[2]
            room = [torch.empty(size + 1, dtype=CDT[prec], device="cuda") for _ in range(3)]
            x, X, y = (r[1:].view(shape) for r in room)
            assert x.data_ptr() % 16 == 8
            torch.view_as_real(x).uniform_(-1, 1)
            ref = torch.fft.fft(x.to(torch.complex128), dim=dim)
            p.forward(x, out=X)
            p.backward(X, out=y)
            torch.cuda.synchronize()
            assert p.device_status() == 0
            assert rel(X, ref) <= TOL[prec] and rel(y, x.to(torch.complex128)) <= TOL[prec]
