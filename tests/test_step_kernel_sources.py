"""Step kernels may start before their predecessor in the stream has ended (programmatic
launches), so the arrays that step kernels write are not declared read-only in them."""
import glob
import os
import re

from paper_2009_12279_gb300 import build

# written on the host's request only, never by a step kernel
UNCHANGED = {"entries", "seg_begin", "seg_flag"}


def _closing(src, i, a, b):
    """Index behind the bracket that closes the one at src[i]."""
    depth = 0
    while True:
        depth += (src[i] == a) - (src[i] == b)
        i += 1
        if depth == 0:
            return i


def _functions(qualifier):
    """{name: (parameters, body)} of the CUDA functions with a qualifier."""
    out = {}
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(qualifier, src):
            i = src.index("(", m.end())
            while re.search(r"__\w+__\s*$", src[m.end():i]):  # __launch_bounds__(...) and the like
                i = src.index("(", _closing(src, i, "(", ")"))
            name = re.search(r"(\w+)\s*$", src[m.end():i])
            end = _closing(src, i, "(", ")")
            tail = re.match(r"\s*(const)?\s*\{", src[end:end + 40])
            if name and tail:
                at = end + tail.end() - 1
                out[name.group(1)] = (src[i:end], src[at:_closing(src, at, "{", "}")])
    return out


def _read_only(params):
    return {p.split()[-1].lstrip("*") for p in params.split(",") if "const " in p and "__restrict__" in p
            for p in [p.rstrip(") \n")]}


def test_step_kernels_declare_no_written_array_read_only():
    kernels = {n: _read_only(p) for n, (p, b) in _functions("__global__").items() if "step_wait()" in b}
    assert {"k_lb", "k_fv_cells", "k_fv_tiled", "k_fv_pair", "k_lb_rows", "k_momentum_exchange",
            "k_momentum_exchange_part", "k_body_reduce", "k_body_partials", "k_particle_phase", "k_read"} <= set(kernels)
    assert {n: r - UNCHANGED for n, r in kernels.items() if r - UNCHANGED} == {}


def test_device_functions_of_the_step_declare_none_either():
    # cell_mask and batch_find serve kernels that are launched plainly
    bad = {n for n, (p, _) in _functions("__device__").items() if _read_only(p)}
    assert bad <= {"cell_mask", "batch_find"}
