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
void stream(uint32_t arrays, uint32_t elem, int writes, int aligned16, uint64_t n, int sched,
            uint64_t chunk, uint32_t teams, uint32_t threads, uint64_t smem_base, int reduction,
            int comp_sum, uint32_t stage_bytes, uint64_t* out) {
  const StreamPlan p = stream_plan({152, 232448, 233472, stage_bytes}, {arrays, elem, 0, writes != 0}, false,
                                   aligned16, n, sched, chunk, teams, threads, smem_base,
                                   reduction, comp_sum);
  out[0] = p.stage_chunks;
  out[1] = p.row_bytes;
  out[2] = p.row_stages;
  out[3] = p.smem;
}
int line(uint64_t n, int sched, uint64_t chunk, uint32_t teams, uint32_t threads) {
  return line_plan({152, 232448, 233472, 32768}, true, n, sched, chunk, teams, threads).smem != 0;
}
int tiles(uint64_t stack, uint64_t n, uint64_t nseg, int dot, uint32_t teams, uint32_t threads) {
  return tile_plan({152, 232448, 233472, 32768}, (uint32_t)stack, n, nseg, dot, teams,
                   threads).tiles;
}
int uneven(uint64_t n, int sched, uint32_t teams, uint32_t threads) {
  return overlap_uneven(n, sched, teams, threads, 152);
}
int window(int64_t budget, uint64_t nx, uint64_t ny, int sched, uint64_t chunk, uint32_t teams,
           uint32_t threads) {
  return window_plan({152, 232448, 233472, 32768}, budget, true, nx, ny, sched, chunk, teams,
                     threads).smem != 0;
}
int cols(uint64_t nx, uint64_t ny, uint32_t teams, uint32_t threads) {
  return cols_applies(nx, ny, teams, threads);
}
}
"""


# schedules as plan.h numbers them
STATIC, CHUNKED, DYNAMIC, AUTO, DIST, GUIDED, NONMONO = range(7)

# body -> (arrays, element bytes, whether it reduces, whether by compensated adds)
BODIES = {"axpy": (2, 4, False, False), "axpy_sum": (2, 4, True, True),
          "axpy_i32_sum": (2, 4, True, False), "dot": (2, 4, True, True),
          "load_f32_sum": (1, 4, True, True), "load_f32_max": (1, 4, True, False),
          "load_bf16_sum": (1, 2, True, True), "load_i32": (1, 4, True, False),
          "load_i64": (1, 8, True, False)}


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


def stream(body, n, sched, chunk, teams, threads, stage_bytes=32768, aligned16=True,
           smem_base=None):
    """The form of a streaming loop on a GB300: ("staged", chunks a pass), ("rows",
    (bytes a row, stages)) or ("plain", None)."""
    arrays, elem, red, comp = BODIES[body]
    out = (C.c_uint64 * 4)()
    base = (4096 if red else 0) if smem_base is None else smem_base
    _lib().stream(arrays, elem, int(body.startswith("axpy")), int(aligned16), C.c_uint64(n), sched,
                  C.c_uint64(chunk), C.c_uint32(teams), C.c_uint32(threads), C.c_uint64(base),
                  int(red), int(comp), C.c_uint32(stage_bytes), out)
    if out[0]:
        return "staged", out[0]
    if out[1]:
        return "rows", (out[1], out[2])
    return "plain", None


def line(n, sched, chunk, teams, threads):
    """Whether a 1-D stencil outside the staged form goes by lanes' pieces."""
    return bool(_lib().line(C.c_uint64(n), sched, C.c_uint64(chunk), C.c_uint32(teams),
                            C.c_uint32(threads)))


def tiles(n, nseg, teams, threads, single_dot=False, stack=4096):
    """Tiles of a generic launch's ring; 0: the plain form."""
    return _lib().tiles(C.c_uint64(stack), C.c_uint64(n), C.c_uint64(nseg), int(single_dot),
                        C.c_uint32(teams), C.c_uint32(threads))


def uneven(n, sched, teams, threads):
    """Whether the region kernel's 2-D stencil goes without launch overlap."""
    return bool(_lib().uneven(C.c_uint64(n), sched, C.c_uint32(teams), C.c_uint32(threads)))


def window(nx, ny, sched, chunk, teams, threads, budget=232448 - 2048):
    """Whether a 2-D stencil that none of the forms before takes goes by block windows."""
    return bool(_lib().window(C.c_int64(budget), C.c_uint64(nx), C.c_uint64(ny), sched,
                              C.c_uint64(chunk), C.c_uint32(teams), C.c_uint32(threads)))
