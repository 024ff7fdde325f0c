"""Radix sequences of the smooth lengths in complex128 (AFFT_SMOOTH_PLANS, csrc/fft_stage.cuh): their lines are
bound by the FP64 pipe, where a warp costs the same however many of its lanes have a butterfly.  The FP64
operations a strided tile issues, idle lanes among them, are at most a tenth above those of one pass per
factor (the sequences of the generic kernels)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07933_gb300", "csrc",
                   "fft_stage.cuh")
# FP64 operations of one butterfly (adds, multiplies, fused pairs), without the twiddles between passes
OPS = {2: 4, 3: 14, 4: 16, 5: 36, 6: 40, 8: 56, 9: 100, 10: 92, 12: 104, 15: 178, 16: 168}


def plans(names):
    text = open(SRC).read()
    out = {}
    for name in names:
        m = re.search(r"#define AFFT_SMOOTH_PLANS_%s\(X\)((?:.*\\\n)*.*\n)" % name, text)
        for entry in re.findall(r"X\(([\d, ]+)\)", m.group(1)):
            n, *radices = map(int, entry.split(","))
            assert n not in out
            out[n] = radices
    return out


def basic(n):
    a, r = 0, []
    while n % 2 == 0:
        n, a = n // 2, a + 1
    passes = (a + 3) // 4
    r += [1 << (a // passes + (i < a % passes)) for i in range(passes)]
    for p in (3, 5):
        while n % p == 0:
            n //= p
            r.append(p)
    return r


def issued(n, radices):
    columns = 8
    while 3 * n * columns * 16 > 200 * 1024:
        columns //= 2
    total, ns = 0, 1
    for r in radices:
        warps = -(-columns * (n // r) // 32)
        total += 32 * warps * (OPS[r] + (4 * (r - 1) if ns > 1 else 0))
        ns *= r
    return total


def test_complex128_sequences_issue_no_more_than_one_pass_per_factor():
    f64 = plans(["A", "B", "C", "D", "F64"])
    f32 = plans(["A", "B", "C", "D", "F32"])
    assert sorted(f64) == sorted(f32) and len(f64) == 67
    for table in (f64, f32):
        for n, radices in table.items():
            prod = 1
            for r in radices:
                prod *= r
            assert prod == n
    slow = {n: issued(n, r) / issued(n, basic(n)) for n, r in f64.items() if len(r) > 1}
    assert max(slow.values()) <= 1.1, {n: round(v, 2) for n, v in slow.items() if v > 1.1}
