"""Kernels launched as programmatic dependents start while the kernel before
them still writes.  A pointer that is both const and __restrict__ allows loads
that need not see those writes, and that the compiler may move above the wait;
so such a kernel has one only for arrays that are complete before any step:
the metrics (M) and the inflow profile."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_09926_gb300", "csrc")
FIXED = {"M", "inflow"}


def _sources():
    return {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
            for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def test_dependents_read_what_steps_write_through_plain_pointers():
    seen = set()
    for name, src in _sources().items():
        for kernel in sorted(set(re.findall(r"launch_dep\(\s*(k_\w+)", src))):
            params = re.search(r"__global__[^;{]*?\b" + kernel + r"\s*\(([^{;]*)\)\s*\{", src)
            assert params, (name, kernel)
            fixed = set(re.findall(r"const \w+\*\s*__restrict__\s+(\w+)", params.group(1)))
            assert fixed <= FIXED, (name, kernel, fixed)
            seen.add(kernel)
    assert {"k_timestep", "k_bc_fill", "k_stage_v", "k_stage_d"} <= seen


def test_helpers_of_the_dependents_do_not_bring_it_back():
    src = _sources()
    for name, fn in (("jz_reduce.cu", "timestep_body"), ("jz_grid.cu", "fill_line"), ("jz_grid.cu", "node_value"),
                     ("jz_grid.cu", "axis_block")):
        params = re.search(r"\b" + fn + r"\s*\(([^{;]*)\)\s*\{", src[name])
        assert params, (name, fn)
        assert set(re.findall(r"const \w+\*\s*__restrict__\s+(\w+)", params.group(1))) <= FIXED, (name, fn)
