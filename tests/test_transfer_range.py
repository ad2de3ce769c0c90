"""Which host arrays the transfers hand to a kernel (csrc/transfer.h), compiled for
the host: only whole doubles, aligned, inside one page-locked range."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1505_02037_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "transfer.h"
int main(int argc, char** argv) {
  auto v = [&](int i) { return strtoull(argv[i], nullptr, 0); };
  puts(lbnr::kernel_reaches(v(1), v(2), v(3), v(4)) ? "kernel" : "copy");
}
"""

TOP = 2 ** 64


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("transfer")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + CSRC, str(d / "p.cpp"),
                           "-o", str(d / "p")])
    return str(d / "p")


@pytest.mark.parametrize("p,nbytes,start,size,want", [
    (0x10000, 0x1000, 0x10000, 0x1000, "kernel"),       # the whole allocation
    (0x10008, 0x0ff8, 0x10000, 0x1000, "kernel"),       # its end, 8 bytes off 16
    (0x10000, 8, 0x10000, 0x1000, "kernel"),
    (0x10000, 0x1008, 0x10000, 0x1000, "copy"),         # past the end
    (0x10000, 0x9000, 0x10000, 0x1000, "copy"),         # ends in another registration
    (0x0fff8, 16, 0x10000, 0x1000, "copy"),             # starts before it
    (0x11000, 8, 0x10000, 0x1000, "copy"),
    (0x10004, 8, 0x10000, 0x1000, "copy"),              # misaligned
    (0x10001, 0x800, 0x10000, 0x1000, "copy"),
    (0x10000, 12, 0x10000, 0x1000, "copy"),             # not whole doubles
    (0x10000, 0, 0x10000, 0x1000, "copy"),
    (0x10000, 8, 0, 0, "copy"),                         # no range known
    (0x10000, TOP - 8, 0x10000, 0x1000, "copy"),        # no wrap-around
    (TOP - 0x1000, 0x1000, TOP - 0x1000, 0x1000, "kernel"),
    (TOP - 8, 16, TOP - 0x1000, 0x1000, "copy"),
])
def test_range(program, p, nbytes, start, size, want):
    got = subprocess.check_output([program, str(p), str(nbytes), str(start), str(size)], text=True)
    assert got.strip() == want
