"""Complex128 fused Poisson stage of one-pass lengths (n0 = 2, 4, 8, 16): float-float, converted by a copy."""
import pytest
import torch

from paper_1506_07933_gb300 import afft

pytestmark = pytest.mark.gpu


def exact(f):
    n = f.shape
    k = [torch.fft.fftfreq(m, 1.0 / m, dtype=torch.float64, device="cuda") for m in n[:2]]
    k.append(torch.arange(n[2] // 2 + 1, dtype=torch.float64, device="cuda"))
    kk = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    kk[0, 0, 0] = float("inf")
    return torch.fft.irfftn(torch.fft.rfftn(f) / kk, s=n)


@pytest.mark.parametrize("n0", [2, 4, 8, 16])
@pytest.mark.parametrize("scale", [1.0, 1e40, 1e-40])   # the last two leave float-float range: FP64
def test_one_pass_lengths(n0, scale):
    # 243 x 201 columns: more tiles of eight than resident CTAs, the last one of three columns
    g = torch.Generator(device="cuda").manual_seed(n0)
    f = torch.rand((n0, 243, 400), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    with afft.Plan(f.shape, "r2c", "f64") as p:
        u = p.poisson(f * scale)
        torch.cuda.synchronize()
        assert p.device_status() == 0
    u = u / scale
    ref = exact(f)
    assert ((u - ref).norm() / ref.norm()).item() <= 1e-12


def test_one_pass_stage_keeps_pace():
    """A 16-point stage (one pass) against a 32-point one (two) over the same number of points: in FP64, with
    eight butterflies a tile, it took 873 us, in float-float 224 us (32 points: about 150 us)."""
    ms = {}
    for n0, n1 in ((16, 1024), (32, 512)):
        with afft.Plan((n0, n1, 512), "r2c", "f64") as p:
            f = torch.rand(p.spatial_shape, dtype=torch.float64, device="cuda")
            u = torch.empty_like(f)
            for _ in range(3):
                p.poisson(f, out=u)
            p.timing_begin(9)
            for _ in range(9):
                p.poisson(f, out=u)
            ms[n0] = sorted(r[1] for r in p.timing_end())[4]
    assert ms[16] <= 3 * ms[32], ms
