"""Plans whose stage kernels start before their predecessor ends (programmatic dependent launch): chains of
transforms and Poisson solves on changing inputs, nothing waited for in between, through every kind of
stage kernel.  A stage that read what its predecessor had not yet written would give other bits than
the same calls with a wait after each, and be far from the 64-bit transform."""
import pytest
import torch

from paper_1506_07933_gb300 import afft

pytestmark = pytest.mark.gpu

# against 64 bits: complex64 a few eps sqrt(log2 N), complex128 lines in float-float or FP64
TOL = {"f32": 2e-6, "f64": 1e-12}

# kind, shape, forward kernels (N2, N1, N0)
CASES = [
    ("c2c", (40, 36, 48), ("k_contig", "k_strided_pipe", "k_strided_pipe")),
    # odd rows of odd length, in place: neighbouring tiles share 128-byte lines
    ("r2c", (48, 75, 96), ("k_r2c", "k_strided", "k_strided_pipe_rp")),
    ("c2c", (27, 45, 81), ("k_contig", "k_strided", "k_strided")),
    ("r2c", (24, 360, 500), ("k_r2c", "k_strided_pipe_rp", "k_strided_pipe")),
    # generic kernels, on a strided and on the contiguous axis
    ("c2c", (6, 1080, 25), ("k_contig", "k_strided", "k_strided_pipe")),
    ("r2c", (30, 40, 2160), ("k_r2c", "k_strided_pipe_rp", "k_strided_pipe")),
    ("c2c", (4, 9, 8192), ("k_strided+k_fourstep", "k_strided_pipe", "k_strided_pipe")),
    # several waves of CTAs per stage
    ("r2c", (256, 256, 256), ("k_r2c", "k_strided_pipe_rp", "k_strided_pipe")),
]


def fields(plan, count):
    g = torch.Generator(device="cuda").manual_seed(7)
    out = []
    for _ in range(count):
        x = torch.empty(plan.spatial_shape, dtype=plan.spatial_dtype, device="cuda")
        (torch.view_as_real(x) if x.is_complex() else x).uniform_(-1, 1, generator=g)
        out.append(x)
    return out


def rel(a, ref):
    a = a.to(ref.dtype)
    return (torch.linalg.vector_norm(a - ref) / torch.linalg.vector_norm(ref)).item()


@pytest.mark.parametrize("kind,shape,kernels", CASES)
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_chained_transforms(kind, shape, kernels, prec):
    with afft.Plan(shape, kind, prec) as p:
        d = p.describe()
        assert d["overlap"] == 1
        if prec == "f32":
            assert tuple(d["stage_kernels_forward"]) == kernels
        xs = fields(p, 3)
        want = []
        for x in xs:
            X = p.forward(x)
            torch.cuda.synchronize()
            y = p.backward(X)
            torch.cuda.synchronize()
            want.append((X, y))
        for x, (X, y) in zip(xs, want):
            wide = x.to(torch.complex128 if x.is_complex() else torch.float64)
            ref = (torch.fft.fftn if kind == "c2c" else torch.fft.rfftn)(wide, dim=(-3, -2, -1))
            assert rel(X, ref) <= TOL[prec] and rel(y, wide) <= TOL[prec]
        buf = torch.empty_like(xs[0])
        X, y = torch.empty_like(want[0][0]), torch.empty_like(buf)
        same = torch.ones((), dtype=torch.bool, device="cuda")
        for i in range(30):
            buf.copy_(xs[i % 3])
            p.backward(p.forward(buf, out=X), out=y)
            same &= (X == want[i % 3][0]).all() & (y == want[i % 3][1]).all()
        assert same.item()
        assert p.device_status() == 0


@pytest.mark.parametrize("shape", [s for k, s, _ in CASES if k == "r2c"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_chained_poisson_solves(shape, prec):
    with afft.Plan(shape, "r2c", prec) as p:
        assert p.describe()["overlap"] == 1
        xs = fields(p, 3)
        want = []
        for x in xs:
            u = p.poisson(x)
            torch.cuda.synchronize()
            v = p.poisson(u)
            torch.cuda.synchronize()
            want.append((u, v))
        buf = torch.empty_like(xs[0])
        u, v = torch.empty_like(buf), torch.empty_like(buf)
        same = torch.ones((), dtype=torch.bool, device="cuda")
        for i in range(30):
            buf.copy_(xs[i % 3])
            p.poisson(p.poisson(buf, out=u), out=v)
            same &= (u == want[i % 3][0]).all() & (v == want[i % 3][1]).all()
        assert same.item()
        assert p.device_status() == 0


@pytest.mark.parametrize("kind,shape", [("r2c", (96, 64, 128)), ("c2c", (64, 75, 90))])
def test_slabs_on_two_streams(kind, shape):
    """Slab by slab (afft_plan_set_l2_chunk) consecutive stages alternate between two streams, ordered by
    events: the same bits as unfused, on inputs that change from call to call."""
    with afft.Plan(shape, kind, "f32") as p:
        xs = fields(p, 3)
        want = [(X, p.backward(X)) for X in [p.forward(x) for x in xs]]
        torch.cuda.synchronize()
        p.set_l2_chunk(shape[0] // 8 * shape[1] * p.spectral_shape[-1] * 8)
        assert p.describe()["l2_slab_planes"] == shape[0] // 8
        buf = torch.empty_like(xs[0])
        X, y = torch.empty_like(want[0][0]), torch.empty_like(buf)
        same = torch.ones((), dtype=torch.bool, device="cuda")
        for i in range(30):
            buf.copy_(xs[i % 3])
            p.backward(p.forward(buf, out=X), out=y)
            same &= (X == want[i % 3][0]).all() & (y == want[i % 3][1]).all()
        assert same.item()
