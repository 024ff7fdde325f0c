"""Kernels that start before their predecessor in the stream has finished (stage_begin, csrc/fft_access.cuh)
read data that changes during their lifetime: none of their pointers but the tables that plan creation
writes may be `__restrict__`, which would allow non-coherent loads."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07933_gb300", "csrc")
TABLES = {"tw", "twr", "post_tw", "wn"}


def closing(text, at, pair):
    """Index just past the bracket that closes the one at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced " + pair)


def kernels():
    """(name, parameter list, body) of every __global__ function of the sources."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+", text):
            at = m.end()
            bounds = re.match(r"__launch_bounds__\s*\(", text[at:])
            if bounds:
                at = closing(text, at + bounds.end() - 1, "()")
            name = re.match(r"\s*(\w+)\s*\(", text[at:])
            end = closing(text, at + name.end() - 1, "()")
            body = text.index("{", end)
            yield name.group(1), text[at + name.end():end - 1], text[body:closing(text, body, "{}")]


def test_overlapped_kernels_have_no_restrict_data():
    seen = set()
    for name, params, body in kernels():
        if "stage_begin()" not in body:
            continue
        seen.add(name)
        for p in params.split(","):
            if "__restrict__" in p:
                assert re.search(r"(\w*)\s*$", p).group(1) in TABLES, (name, p.strip())
    assert {"k_strided", "k_contig", "k_r2c", "k_c2r", "k_fourstep", "k_strided_pipe", "k_strided_pipe_rp",
            "k_poisson_pipe", "k_poisson_mult", "k_scale"} <= seen


def test_no_kernel_triggers_its_dependents_early():
    """CTAs launched while the previous kernel still fills the GPU crowd onto the SMs with room (stage_begin)."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "griddepcontrol.launch_dependents;" not in re.sub(r"//[^\n]*", "", open(path).read()), path
