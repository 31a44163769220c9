"""CPU check of the kernels' sources: the read-only load path (__ldg,
ld.global.nc, const __restrict__ parameters) is for data that nothing writes
from a kernel's start to its end.  A kernel launched with launch_dependent runs
while its predecessor still writes its inputs, so there only links, clover and
SAP's block-ordered copies may go through it; spinors, CG vectors, activations
and what a kernel updates in place take ordinary loads."""
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
    # the arrays that reach the read-only path: the links of a hop, SAP's clover copy and the kernel that makes it
    fixed = {"dslash_impl.cuh": {"lp"}, "sap.cu": {"src", "clb"}}
    for n in names:
        text = code(n)
        if n == "core.cuh":
            # the definitions, then the links' and the clover term's loads, whose callers choose
            text, k = re.subn(r"return FIXED \? __ldg\(p\) : \*p;|T ld_fixed\(const T\* p\)", "", text)
            assert k == 2
            text, k = re.subn(r"struct GaugeIO;.*?inline size_t gauge_link_bytes|struct CloverIO;.*?inline size_t clover_site_bytes",
                              "", text, flags=re.S)
            assert k == 2
        assert "__ldg" not in text and "ld.global.nc" not in text and "ld<FIXED>" not in text, n
        if n in dependent:
            assert "__restrict__" not in text, n
            assert set(re.findall(r"ld_fixed\((\w+)", text)) == fixed.get(n, set()), n


def test_first_launch_behind_a_load_is_plain():
    """Links and clover are read-only data for the hopping kernels because the
    launch behind a load waits for all of it."""
    api, impl = code("api.cu"), code("dslash_impl.cuh")
    for entry in ("lqcd_gauge_load", "lqcd_clover_compute"):
        body = api[api.index("lqcd_status %s(" % entry):]
        assert "c->links_new = 1" in body[:body.index("\n}\n")], entry
    assert "A.plain = c->links_new" in api
    assert impl.count("launch_dependent(") == impl.count("if (A.plain) {") == 2
