"""Loads in kernels that may start while the launch before them still writes (griddepcontrol): PTX lets the
non-coherent path (__ldg, or a const __restrict__ parameter that the compiler turns into it) read only data
that no one writes during the kernel's lifetime, which there includes the writes of the launch before. So
__ldg takes unit tables and masks only, and no such kernel has a const __restrict__ parameter. A stale value
would show as a wrong time step or state on some runs only, so the sources are checked."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_09272_gb300", "csrc")
WRITTEN_BY_NO_KERNEL = {"a.units", "a.tiles", "a.solid"}


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*(?:\([^()]*\)[^()]*)*\))*\)\s*)?(\w+)\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, b = text[m.end():i - 1], text.index("{", i)
        depth, j = 1, b + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), params, text[b:j]


def test_ldg_reads_only_what_no_kernel_writes():
    seen = 0
    for name, text in sources():
        for m in re.finditer(r"__ldg\(([^;]*?)\)", text):
            seen += 1
            base = m.group(1).split("+")[0].strip()
            assert base in WRITTEN_BY_NO_KERNEL, (name, m.group(0))
    assert seen >= 4


def test_kernels_that_start_early_have_no_read_only_parameters():
    early = set()
    for name, text in sources():
        for kernel, params, body in kernels(text):
            if "pdl_wait()" in body:
                early.add(kernel)
                for p in params.split(","):
                    assert not ("const" in p.split("*")[0] and "__restrict__" in p), (name, kernel, p)
                assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", body), (name, kernel)
    assert {"stage_kernel", "tile_kernel", "pack_kernel", "unpack_kernel"} <= early
