"""CPU check of the kernels' sources: the read-only load path (__ldg,
ld.global.nc, const __restrict__ parameters) is for data that nothing writes
from a kernel's start to its end.  A kernel launched with launch_dependent runs
while its predecessor still writes its inputs, so the shared loads (core.cuh),
the hopping kernels, the BLAS kernels and the network take ordinary loads."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1103_1363_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


def test_dependent_launches_take_ordinary_loads():
    names = sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh")))
    dependent = [n for n in names if re.search(r"launch_dependent\(|griddepcontrol", code(n))]
    assert {"core.cuh", "dslash_impl.cuh", "blas.cu", "net.cu", "sap.cu"} <= set(dependent)
    for n in names:
        text = code(n)
        if n == "core.cuh":  # the one definition
            text, k = re.subn(r"T ld_fixed\(const T\* p\)\s*\{\s*return __ldg\(p\);\s*\}", "", text)
            assert k == 1
        assert "__ldg" not in text and "ld.global.nc" not in text, n
        if n in dependent:
            assert "__restrict__" not in text, n
            # SAP's block-ordered clover term, complete before the chain of launches, and the copy that makes it
            uses = re.findall(r"ld_fixed\((\w+)", text)
            assert uses == (["src", "clb"] if n == "sap.cu" else []), (n, uses)
