"""Which fields the operators take in place, on the host.

A kernel may only be given memory that it reaches, aligned to the field's
elements, with all of the field inside one allocation. The decision is that of
csrc/host_common.h, compiled unchanged by the host compiler; a field that it
turns down goes through a copy, which the driver checks. (A buffer that ends
early is not tried on a GPU.)
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_05970_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "host_common.h"
using namespace fftg;

int main(int argc, char** argv) {
    BufferRange r;
    r.here = std::atoi(argv[1]) != 0;
    r.base = (uintptr_t)std::strtoull(argv[2], nullptr, 0);
    r.size = (size_t)std::strtoull(argv[3], nullptr, 0);
    const void* p = (const void*)(uintptr_t)std::strtoull(argv[4], nullptr, 0);
    std::printf("%d\n", usable_in_place(r, p, (size_t)std::strtoull(argv[5], nullptr, 0), (size_t)std::atoi(argv[6])));
}
"""

BASE, TOP = 0x7f0000000000, 2 ** 64


@pytest.fixture(scope="module")
def decide(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("ranges")
    (d / "t.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return lambda *a: subprocess.run([str(d / "t")] + [str(x) for x in a], capture_output=True, text=True,
                                     check=True).stdout.strip() == "1"


@pytest.mark.parametrize("here,base,size,p,nbytes,es,want", [
    (1, BASE, 1296, BASE, 1296, 8, True),               # a whole allocation
    (1, BASE, 1295, BASE, 1296, 8, False),              # a byte short
    (1, BASE, 4096, BASE + 2800, 1296, 8, True),        # up to the allocation's end
    (1, BASE, 4096, BASE + 2808, 1296, 8, False),       # an element past it
    (1, BASE, 4096, BASE + 4096, 1296, 8, False),       # behind it
    (1, BASE, 4096, BASE - 8, 1296, 8, False),          # in front of it
    (1, BASE, 4096, BASE + 4, 648, 4, True),
    (1, BASE, 4096, BASE + 4, 1296, 8, False),          # not aligned to its elements
    (1, BASE, 4096, BASE + 2, 648, 4, False),
    (0, BASE, 4096, BASE, 1296, 8, False),              # not this device's memory
    (1, 0, 0, BASE, 1296, 8, False),                    # allocation not known
    (1, TOP - 4096, 4095, TOP - 1296, 1296, 8, False),  # the end of the address space
    (1, TOP - 4096, 4096, TOP - 1296, 1296, 8, True),
    (1, TOP - 4096, 4096, TOP - 1288, 1296, 8, False),
])
def test_in_place(decide, here, base, size, p, nbytes, es, want):
    assert decide(here, base, size, p, nbytes, es) is want
