"""Rule of the kernels that a step launches while their predecessor still runs
(chain_begin in lbgb_internal.cuh): what the predecessor writes is not
read-only for their lifetime, so the sources hold no non-coherent load
(__ldg, ld.global.nc), and no such kernel has a const __restrict__ parameter,
from which the compiler derives one."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_04080_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def kernels(src):
    """(name, parameters, text up to the next kernel) of each kernel."""
    starts = [m.start() for m in re.finditer(r"__global__ void", src)] + [len(src)]
    for a, b in zip(starts, starts[1:]):
        m = re.search(r"(\bk\d?_\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", src[a:b])
        yield m.group(1), m.group(2), src[a:b]


def test_no_non_coherent_loads():
    for name, src in sources():
        assert "__ldg" not in src and "global.nc" not in src, name


def test_chained_kernels():
    found = set()
    for name, src in sources():
        launched = set(re.findall(r"launch_after\(\s*(\w+)", src)) - {"void"}
        for kernel, params, text in kernels(src):
            if kernel not in launched:
                continue
            found.add(kernel)
            body = text[text.index("{") + 1 :].split(";")[0]
            assert "chain_begin()" in body, "%s: chain_begin is not the first statement" % kernel
            for p in params.split(","):
                assert not ("const" in p and "__restrict__" in p), (kernel, p)
    assert {"k_moments", "k_bounce_links", "k_lean", "k_density", "k_virtual", "k_remap_create"} <= found
