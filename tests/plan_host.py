"""The library's rules for the form of a launch (csrc/plan.h), compiled for the
host by g++ and called through ctypes: the same code the library runs."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

from paper_2106_03219_gb300 import build_lib

SOURCE = r"""
#include "plan.h"
using namespace rt;
extern "C" {
int cols(uint64_t nx, uint64_t ny, uint32_t teams, uint32_t threads) {
  return cols_applies(nx, ny, teams, threads);
}
}
"""


@functools.lru_cache(maxsize=None)
def _lib():
    d = tempfile.mkdtemp()
    src, so = os.path.join(d, "plan.cpp"), os.path.join(d, "plan.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", build_lib.CSRC, src, "-o",
                    so], check=True)
    return C.CDLL(so)


def cols(nx, ny, teams, threads):
    """Whether a schedule(auto) 2-D stencil off the tensor tiles walks strips of columns."""
    return bool(_lib().cols(C.c_uint64(nx), C.c_uint64(ny), C.c_uint32(teams), C.c_uint32(threads)))
