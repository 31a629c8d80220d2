"""Kernels that start while the kernel before them still runs must not claim
that nothing writes what they read: a read-only load (__ldg, or a pointer
parameter that is const and __restrict__) may be moved above the wait for the
kernel before.  Checked on the sources, for every kernel launched so; the
instance descriptors, which no kernel writes, may be read in any way."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_6238_gb300", "csrc")
TEXT = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f, encoding="utf-8").read())
        for f in glob.glob(os.path.join(CSRC, "*.cu*"))}
ALL = "\n".join(TEXT.values())
KERNELS = sorted(set(re.findall(r"launch_early\(\s*(\w+)", ALL)))


def test_the_kernels_are_found():
    assert {"tile_kernel", "stash_kernel", "drive_kernel", "adjoint_A"} <= set(KERNELS)


@pytest.mark.parametrize("name", KERNELS)
def test_parameters(name):
    m = re.search(r"__global__[^;{]*?\b%s\s*\(([^)]*)\)\s*\{" % name, ALL)
    assert m, name
    for p in m.group(1).split(","):
        if "const" in p.split("*")[0] and "__restrict__" in p:
            assert re.match(r"\s*const InstDev\*", p), p.strip()


def test_no_read_only_loads():
    for name, text in TEXT.items():
        assert "__ldg(" not in text, name
