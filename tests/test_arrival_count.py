"""The arrival count of the grid-wide barrier (csrc/common.cuh, compiled for the host): a CTA leaves
barrier k only when all G CTAs have arrived at it, also where the 32-bit count wraps."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2511_06788_gb300 import build as B

SRC = r"""
#include "common.cuh"
extern "C" int reached(unsigned count, unsigned target) { return opevo::count_reached(count, target); }
"""


@pytest.fixture(scope="module")
def reached(tmp_path_factory):
    d = tmp_path_factory.mktemp("count")
    src, so = os.path.join(d, "count_host.cu"), os.path.join(d, "count_host.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-I", B.INCLUDE,
                    "-I", B.CSRC, "-shared", "-o", so, src], check=True)
    lib = C.CDLL(so)
    lib.reached.argtypes = [C.c_uint, C.c_uint]
    return lib.reached


@pytest.mark.parametrize("G", [2, 117, 152])
def test_a_barrier_opens_when_all_have_arrived(reached, G):
    start = 2**32 // G - 3  # barriers before the wrap
    for k in range(start, start + 7):
        target = (k + 1) * G % 2**32
        for here in range(G + 1):  # arrivals at barrier k; the others are there already or at k + 1
            assert bool(reached((k * G + here) % 2**32, target)) == (here == G)
        for later in range(G):  # a slow CTA looks while others arrive at the next barrier
            assert reached(((k + 1) * G + later) % 2**32, target)
