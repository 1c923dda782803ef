"""Pointer qualifiers that promise more than a kernel's launches keep, read from the
sources: __restrict__ on buffers that may be one, and on inputs that another kernel
may still be writing when this one starts (the compiler may then load them through the
read-only path, which is not ordered by a wait inside the kernel)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_11027_gb300", "csrc")


def functions():
    """(name, parameter list, body) of every function in the CUDA sources."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        for m in re.finditer(r"\b(\w+)\(([^;{}()]*(?:\([^()]*\)[^;{}()]*)*)\)\s*\n\{\n", text):
            end = text.index("\n}\n", m.end() - 1)
            yield m.group(1), m.group(2), text[m.end():end]


def named(name):
    found = [f for f in functions() if f[0] == name]
    assert found, name
    return found


def test_resident_pools_may_be_one_buffer():
    for name in ("k_batch_resident", "resident_domain", "resident_rows"):
        for _, params, _ in named(name):
            for p in params.split(","):
                if re.search(r"\b(pool_in|pool_out|A0|B0)\b", p):
                    assert "__restrict__" not in p, (name, p)


def test_early_launched_kernels_read_by_ordinary_loads():
    early = [f for f in functions() if re.search(r"\bpdl_begin\(\);", f[2])]
    assert len(early) >= 2
    called = [f for name in ("gather", "store_psi") for f in named(name)]
    for name, params, body in early + called:
        assert "__restrict__" not in params, name
        assert "__ldg(" not in body and "ld.global.nc" not in body, name
