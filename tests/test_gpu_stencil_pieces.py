"""GPU parity: the 2-D stencil on grids and team blocks of any length: a team's
whole block in shared memory, or (the budget too small for it) lanes' pieces
staged with the rows above and below (static, static(c), dynamic(c),
nonmonotonic), and strips of columns (auto on odd grids).

Grids put rows at every place of a 16-byte unit, rows shorter than a staged
row and than the stencil, boundary points everywhere in a row, array ends inside
a unit, and arrays off 16 bytes; bit-exact against the oracle, the elements
around the output untouched."""
import numpy as np
import pytest

import oracle as O
from paper_2106_03219_gb300 import inputs
from paper_2106_03219_gb300 import omprt as R
from gpu_helpers import bits32, dev, host

pytestmark = pytest.mark.gpu

GRIDS = [(1, 4099), (4099, 1), (2051, 2), (1400, 3), (900, 5), (301, 33), (130, 127), (129, 514),
         (67, 1001), (255, 256), (40, 4095), (33, 4100)]
SCHEDS = [(R.SCHED_STATIC, 0), (R.SCHED_STATIC_CHUNKED, 9), (R.SCHED_STATIC_CHUNKED, 32), (R.SCHED_STATIC_CHUNKED, 61),
          (R.SCHED_STATIC_CHUNKED, 300), (R.SCHED_DYNAMIC, 33), (R.SCHED_DYNAMIC, 64),
          (R.SCHED_NONMONOTONIC, 100)]


def _check(rt, ny, nx, sched, chunk, G, T, off=0):
    import torch
    a = inputs.grid_f32(ny, nx, 7)
    n = ny * nx
    buf = torch.zeros(n + 8, device="cuda")
    buf[off:off + n] = dev(a).view(-1)
    out = torch.full((n + 8,), -7.0, device="cuda")
    rt.launch_region(R.loop_desc(R.BODY_STENCIL2D5, n=n, x=buf[off:off + n], out=out[off:off + n],
                                 nx=nx, ny=ny), sched, chunk, G, T)
    got = host(out)
    assert np.array_equal(bits32(got[off:off + n]), bits32(O.stencil2d5(a)).reshape(-1)), (ny, nx)
    assert (got[:off] == -7.0).all() and (got[off + n:] == -7.0).all()


@pytest.mark.parametrize("sched,chunk", SCHEDS)
@pytest.mark.parametrize("G,T", [(1, 32), (3, 96), (2, 256), (1, 512), (4, 1024)])
@pytest.mark.parametrize("budget", [16, 226 * 1024])  # pieces; windows where they fit
def test_pieces_and_windows_bit_exact(rt, sched, chunk, G, T, budget):
    rt.set_stencil_stage_bytes(budget)
    try:
        for ny, nx in GRIDS:
            _check(rt, ny, nx, sched, chunk, G, T)
            if nx == 514 or nx == 1001:  # small blocks: short windows, empty threads
                _check(rt, ny, nx, sched, chunk, 40 * G, T)
            _check(rt, ny, nx, sched, chunk, 2 * G, T, 4)  # off 32 bytes, on 16
    finally:
        rt.set_stencil_stage_bytes(226 * 1024)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("G,T", [(1, 32), (7, 256), (152, 1024), (608, 256)])
def test_cols_bit_exact(rt, G, T):
    for ny, nx in GRIDS + [(1, 1), (2, 2), (3, 63), (9, 64), (8, 65), (700, 129), (1023, 1025)]:
        _check(rt, ny, nx, R.SCHED_AUTO, 0, G, T)
    for off in (1, 2, 3):  # rows of whole units, arrays that do not start on one
        _check(rt, 100, 128, R.SCHED_AUTO, 0, G, T, off)
    assert rt.sync_status() == 0


def test_runtime_team_counts_and_budget_off(rt):
    """The runtime's own team count on an odd and an even grid, with the form
    and with the stencil budget off."""
    for ny, nx in ((1203, 1501), (1100, 1024)):
        for sched, chunk in SCHEDS:
            _check(rt, ny, nx, sched, chunk, 40, 256)
    rt.set_stencil_stage_bytes(0)
    try:
        for sched, chunk in SCHEDS:
            _check(rt, 403, 501, sched, chunk, 0, 0)
    finally:
        rt.set_stencil_stage_bytes(226 * 1024)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("sched,chunk", SCHEDS)
@pytest.mark.parametrize("G,T", [(1, 32), (3, 96), (2, 256), (3, 1024)])
def test_stencil1d_pieces_bit_exact(rt, sched, chunk, G, T):
    import torch
    for n in (1, 2, 33, 4100, 40_961, 300_006, (1 << 20) + 3):
        for off in (0, 4):
            a = inputs.f32_uniform01(n + 8, 4)
            out = torch.full((n + 8,), -7.0, device="cuda")
            rt.launch_region(R.loop_desc(R.BODY_STENCIL1D3, n=n, x=dev(a)[off:off + n],
                                         out=out[off:off + n]), sched, chunk, G, T)
            got = host(out)
            want = O.stencil1d3(np.ascontiguousarray(a[off:off + n]))
            assert np.array_equal(bits32(got[off:off + n]), bits32(want)), (n, off)
            assert (got[:off] == -7.0).all() and (got[off + n:] == -7.0).all()
    assert rt.sync_status() == 0
