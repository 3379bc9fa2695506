"""Shared-memory arrays that a kernel reads 16 bytes at a time carry their
alignment in their declaration: without it the compiler may place them on a
4-byte boundary whenever another shared variable is added."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_03425_gb300", "csrc")
WIDE = re.compile(r"reinterpret_cast<(?:const )?(?:float4|uint4|int4|ulonglong2|double2) \*>\(&(\w+)\[")


def test_wide_reads_have_declared_alignment():
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = open(os.path.join(CSRC, f)).read()
        for kernel in src.split("__global__")[1:]:
            for name in set(WIDE.findall(kernel)):
                seen += 1
                decl = re.search(r"__shared__[^;]*\b%s\[[^;]*;" % name, kernel)
                # or a reference to the member of an aligned struct
                alias = re.search(r"&%s = \w+_\.v\b" % name, kernel)
                assert alias or (decl and "__align__(16)" in decl.group(0)), "%s: %s" % (f, name)
    assert seen > 0
