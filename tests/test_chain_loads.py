"""The kernels that may start before the one before them has finished read memory with ordinary loads only.

A kernel launched with programmatic serialisation can be resident while the buffers it will read are still being
written; the wait inside it orders ordinary loads, and not those of the read-only path (`__ldg`, `ld.global.nc`,
and what the compiler makes of a kernel's `const __restrict__` parameters).  That such a load went wrong was never
seen and cannot be provoked, so the sources are looked at."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_12292_gb300", "csrc")


def _sources():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
    # without comments
    return {f: re.sub(r"//[^\n]*|/\*.*?\*/", "", open(f).read(), flags=re.S) for f in files}


def test_no_read_only_loads():
    for f, s in _sources().items():
        assert not re.search(r"__ldg\w*\s*\(|\.nc\.|__ldcg?s?\s*\(\s*\(const", s), f


def test_chained_kernels_take_no_restrict_parameters():
    for f, s in _sources().items():
        kernels = re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\((.*?)\)\s*\{(.*?)\n\}",
                             s, flags=re.S)
        assert len(kernels) == len(re.findall(r"__global__", s)), f
        for name, params, body in kernels:
            if "launch_wait" in body:
                assert "__restrict__" not in params, (f, name)
