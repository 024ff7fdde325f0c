"""Performance cases: what a user of this library has it do, through its public entry points.

A pass is what a spectral code does once per step: a forward and a backward transform of one plan
("transform"), one periodic Poisson solve ("poisson"), or the forward and backward transforms of a
set of cubic fields of uneven sizes, replayed as one CUDA graph ("graph") or run as one persistent
launch per direction ("persistent").  Inputs and plans are what a program holds before the call.
"""
import math

import torch

from paper_1506_07933_gb300 import afft, synth

# edge lengths of the uneven workload and of the served Poisson solves
UNEVEN = (48, 64, 96, 120, 128, 160, 256)
SERVED = (64, 128, 192, 256, 384, 512)


def _t(name, kind, prec, n0, n1, n2, batch=1):
    return {"name": name, "op": "transform", "kind": kind, "prec": prec, "n0": n0, "n1": n1, "n2": n2, "batch": batch}


def listed():
    return [
        # a small accuracy-first transform in a latency-bound loop: three short launches each way
        _t("c2c_32_f64", "c2c", "f64", 32, 32, 32),
        # the smallest request of the Poisson server, alone on the GPU
        {"name": "poisson_64_f32", "op": "poisson", "prec": "f32", "n0": 64, "n1": 64, "n2": 64, "batch": 1},
        # a batch of equal fields behind one plan (what the server forms from waiting requests)
        _t("r2c_128_f32_batch32", "r2c", "f32", 128, 128, 128, 32),
        # the ordinary real field, and the headline size in both precisions
        _t("r2c_256_f32", "r2c", "f32", 256, 256, 256),
        _t("r2c_512_f32", "r2c", "f32", 512, 512, 512),
        _t("r2c_512_f64", "r2c", "f64", 512, 512, 512),
        # the largest: 8 GB of complex data in, 8 GB out
        _t("c2c_1024_f32", "c2c", "f32", 1024, 1024, 1024),
        # physical grids that are not powers of two: a cube of threes, and uneven real fields
        _t("c2c_243_f32", "c2c", "f32", 243, 243, 243),
        _t("r2c_320x300x500_f32", "r2c", "f32", 320, 300, 500),
        _t("r2c_180x200x216_f64", "r2c", "f64", 180, 200, 216),
        # 200 real fields of uneven sizes, every pass a replay of one captured graph per direction
        {"name": "uneven_200_graph", "op": "uneven", "engine": "graph", "fields": 200, "sizes_seed": 200},
        # the same set as one persistent launch per direction
        {"name": "uneven_200_persistent", "op": "uneven", "engine": "persistent", "fields": 200, "sizes_seed": 200},
    ]


def _smooth(rng, lo, hi, even):
    """A length with prime factors 2, 3, 5, spread over the logarithm of lo .. hi."""
    sizes = [n for n in range(lo, hi + 1) if not (even and n % 2) and _is_smooth(n)]
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sizes, key=lambda n: abs(math.log(n / want)))


def _is_smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    what = rng.random()
    if what < 0.15:
        return {"op": "uneven", "engine": rng.choice(["graph", "persistent"]), "fields": int(8 * 25 ** rng.random()),
                "sizes_seed": rng.randrange(1 << 20)}
    prec = "f32" if rng.random() < 0.65 else "f64"
    if what < 0.35:
        n = rng.choice([s for s in SERVED if prec == "f32" or s < 512])
        batch = rng.choice([1, 2, 4, 8]) if n <= 192 else 1
        return {"op": "poisson", "prec": prec, "n0": n, "n1": n, "n2": n, "batch": batch}
    kind = rng.choice(["c2c", "r2c"])
    if rng.random() < 0.25:   # cubes of the usual lengths
        n = rng.choice([32] + list(UNEVEN) + [192, 384])
        shape = (n, n, n)
    else:                     # any lengths the library takes, odd ones among them
        most = 2 ** 26.5 if prec == "f32" else 2 ** 23
        while True:
            shape = (_smooth(rng, 16, 640, False), _smooth(rng, 16, 640, False), _smooth(rng, 16, 640, kind == "r2c"))
            if math.prod(shape) <= most:
                break
    points = math.prod(shape)
    batch = rng.choice([2, 5, 16]) if points <= 1 << 20 and rng.random() < 0.5 else 1
    return {"op": "transform", "kind": kind, "prec": prec, "n0": shape[0], "n1": shape[1], "n2": shape[2], "batch": batch}


def _sizes(case):
    """Counts per cubic size of an uneven set."""
    sizes = synth.batched_sizes(case["fields"], seed=case["sizes_seed"], choices=UNEVEN)
    return [(n, sizes.count(n)) for n in UNEVEN if n in sizes]


def _real_fields(shape, batch, dtype, seed):
    """Sums of random Fourier modes plus 1e-3 noise, the fields a spectral code transforms."""
    out = torch.empty((batch,) + tuple(shape), dtype=dtype, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    if math.prod(shape) <= 1 << 21 and batch > 1:   # many small fields: one mode sum, each with its own noise and size
        f = synth.random_mode_field_torch(shape, seed, n_modes=16, noise=0.0)
        amp = torch.rand(batch, generator=g, device="cuda", dtype=torch.float64) + 0.5
        for b in range(batch):
            out[b] = f * amp[b] + 1e-3 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    else:
        for b in range(batch):
            out[b] = synth.random_mode_field_torch(shape, seed + b, n_modes=16, noise=1e-3)
    return out


def _input(case, seed):
    shape, batch = (case["n0"], case["n1"], case["n2"]), case["batch"]
    if case["op"] == "transform" and case["kind"] == "c2c":
        x = torch.empty((batch,) + shape, dtype=torch.complex64 if case["prec"] == "f32" else torch.complex128,
                        device="cuda")
        g = torch.Generator(device="cuda").manual_seed(seed)
        torch.view_as_real(x).uniform_(-1.0, 1.0, generator=g)
        return x
    return _real_fields(shape, batch, torch.float32 if case["prec"] == "f32" else torch.float64, seed)


def prepare(case, seed):
    if case["op"] == "uneven":
        plans, xs = [], []
        for i, (n, count) in enumerate(_sizes(case)):
            plans.append(afft.Plan((n, n, n), "r2c", "f32", batch=count))
            xs.append(_real_fields((n, n, n), count, torch.float32, seed + 1000 * i).reshape(plans[-1].spatial_shape))
        Xs = [torch.empty(p.spectral_shape, dtype=p.spectral_dtype, device="cuda") for p in plans]
        ys = [torch.empty_like(x) for x in xs]
        engine = (afft.Multi if case["engine"] == "graph" else afft.Queue)(plans)
        return {"op": "uneven", "engine": engine, "plans": plans, "xs": xs, "Xs": Xs, "ys": ys}
    kind = case["kind"] if case["op"] == "transform" else "r2c"
    plan = afft.Plan((case["n0"], case["n1"], case["n2"]), kind, case["prec"], batch=case["batch"])
    x = _input(case, seed)
    state = {"op": case["op"], "plan": plan, "x": x, "y": torch.empty_like(x)}
    if case["op"] == "transform":
        state["X"] = torch.empty(plan.spectral_shape, dtype=plan.spectral_dtype, device="cuda")
    return state


def run(state):
    if state["op"] == "uneven":
        state["engine"].forward(state["xs"], state["Xs"])
        state["engine"].backward(state["Xs"], state["ys"])
        return {"spectra": state["Xs"], "fields": state["ys"]}
    plan = state["plan"]
    if state["op"] == "poisson":
        return {"u": plan.poisson(state["x"], out=state["y"])}
    X = plan.forward(state["x"], out=state["X"])
    return {"spectrum": X, "field": plan.backward(X, out=state["y"])}


def _one(kind, prec, shape, batch):
    """Bytes of one array of each side and flops (5 N log2 N, half of that for real fields)."""
    points = math.prod(shape) * batch
    real = 4 if prec == "f32" else 8
    bins = points if kind == "c2c" else points // shape[2] * (shape[2] // 2 + 1)
    flops = (5.0 if kind == "c2c" else 2.5) * points * math.log2(max(2, math.prod(shape)))
    return points * real * (2 if kind == "c2c" else 1), bins * real * 2, flops


def work(case):
    if case["op"] == "uneven":
        parts = [_one("r2c", "f32", (n, n, n), count) for n, count in _sizes(case)]
        return {"bytes": sum(2 * (a + b) for a, b, _ in parts), "flops": sum(2 * f for _, _, f in parts)}
    shape = (case["n0"], case["n1"], case["n2"])
    if case["op"] == "poisson":
        a, _, f = _one("r2c", case["prec"], shape, case["batch"])
        return {"bytes": 2 * a, "flops": 2 * f}
    a, b, f = _one(case["kind"], case["prec"], shape, case["batch"])
    return {"bytes": 2 * (a + b), "flops": 2 * f}


def _wavenumbers(n):
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    return torch.where(2 * k > n, k - n, k)


def exact(case, seed):
    """The spectrum from torch.fft in 64 bits; the field that comes back is the input itself."""
    if case["op"] == "uneven":
        spectra, fields = [], []
        for i, (n, count) in enumerate(_sizes(case)):
            x = _real_fields((n, n, n), count, torch.float32, seed + 1000 * i).double()
            fields.append(x)
            spectra.append(torch.fft.rfftn(x, dim=(1, 2, 3)))
        return {"spectra": spectra, "fields": fields}
    x = _input(case, seed)
    x = x.to(torch.complex128 if x.is_complex() else torch.float64)
    if case["op"] == "poisson":
        k0, k1 = _wavenumbers(case["n0"]), _wavenumbers(case["n1"])
        k2 = torch.arange(case["n2"] // 2 + 1, device="cuda", dtype=torch.float64)
        k = k0[:, None, None] ** 2 + k1[None, :, None] ** 2 + k2[None, None, :] ** 2
        k[0, 0, 0] = math.inf
        u = torch.fft.irfftn(torch.fft.rfftn(x, dim=(1, 2, 3)) / k, s=x.shape[1:], dim=(1, 2, 3))
        return {"u": u}
    X = torch.fft.fftn(x, dim=(1, 2, 3)) if case["kind"] == "c2c" else torch.fft.rfftn(x, dim=(1, 2, 3))
    return {"spectrum": X, "field": x}
