"""CPU: what a lane of the 2-D stencil's piece form fetches, enumerated from the
kernel's own index arithmetic (csrc/piece_spans.h) over small grids, every row
position and every piece of a row: no fetch leaves the grid, and every neighbour
of an inner point is fetched.

A grid one column wide would move the span above by up = 4 for nx = 1, and its last
unit would reach past the array's last element: no point needs it, and none is fetched."""
import subprocess

from paper_2106_03219_gb300 import build_lib

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "piece_spans.h"
using namespace rt;

static uint64_t n;
static std::vector<char> have;  // element of the grid fetched into the span at hand
static int bad = 0;
static void fetch(int64_t at, uint32_t bytes, const char* what, uint64_t nx, uint64_t row,
                  uint32_t j0, uint32_t j1) {
  if (at < 0 || bytes == 0 || bytes > 16 || at + bytes / 4 > n || bytes % 4) {
    if (++bad < 20)
      printf("%s nx=%llu n=%llu row=%llu [%u,%u): %lld + %u bytes\n", what,
             (unsigned long long)nx, (unsigned long long)n, (unsigned long long)row, j0, j1,
             (long long)at, bytes);
    return;
  }
  for (uint32_t k = 0; k < bytes / 4; ++k) have[at + k] = 1;
}

template <uint32_t RE>
static void grid(uint64_t nx, uint64_t ny) {
  n = nx * ny;
  const uint32_t sn = (4 - nx % 4) % 4, ss = nx % 4;
  const uint64_t up = piece_up(nx), down = nx - ss;
  for (uint64_t row = 0; row < n; row += RE) {
    const PieceSpans s = piece_spans<RE>(row, n, up, down);
    if (s.ce > 255 || s.ab > 255 || s.be > 255) ++bad;
    for (uint32_t j0 = 0; j0 < RE && row + j0 < n; ++j0)
      for (uint32_t j1 = j0 + 1; j1 <= RE && row + j1 <= n; ++j1) {
        std::vector<char> span[3];
        for (int k = 0; k < 3; ++k) {
          have.assign(n, 0);
          if (k == 1 && j0 == 0 && row > 0) fetch(row - 4, 16, "left", nx, row, j0, j1);
          for (uint32_t u = 0; u <= RE; u += 4) {
            if (u == RE && k != 1 && !(sn | ss)) continue;
            if (k == 0 && (u == RE ? above_edge(RE, j1, sn, s.ab) : above_fetched(u, j0, j1, sn, s.ab)))
              fetch((int64_t)row - (int64_t)up + u, 16, "above", nx, row, j0, j1);
            if (k == 1 && (u == RE ? centre_edge(RE, j1, s.ce) : centre_fetched(u, j0, j1, s.ce)))
              fetch(row + u, unit_bytes(u, s.ce), "centre", nx, row, j0, j1);
            if (k == 2 && (u == RE ? below_edge(RE, j1, ss, s.be) : below_fetched(u, j0, j1, ss, s.be)))
              fetch(row + down + u, unit_bytes(u, s.be), "below", nx, row, j0, j1);
          }
          span[k] = have;
        }
        for (uint64_t i = row + j0; i < row + j1; ++i) {
          const uint64_t r = i / nx, c = i % nx;
          bool ok = span[1][i];
          if (r > 0 && r + 1 < ny && c > 0 && c + 1 < nx)
            ok = ok && span[0][i - nx] && span[1][i - 1] && span[1][i + 1] && span[2][i + nx];
          if (!ok && ++bad < 20)
            printf("not fetched: nx=%llu ny=%llu i=%llu row=%llu [%u,%u)\n", (unsigned long long)nx,
                   (unsigned long long)ny, (unsigned long long)i, (unsigned long long)row, j0, j1);
        }
      }
  }
}

int main() {
  for (uint64_t nx = 1; nx <= 40; ++nx)
    for (uint64_t ny = 1; nx * ny <= 150; ++ny) {
      grid<16>(nx, ny);
      grid<32>(nx, ny);
    }
  printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_fetches_stay_in_the_grid_and_cover_the_points(tmp_path):
    src, exe = tmp_path / "spans.cpp", tmp_path / "spans"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", build_lib.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
