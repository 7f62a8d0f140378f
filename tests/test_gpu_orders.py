"""GPU parity: values and orders that the other tests of the staged forms leave out.

  - infinities, NaN and the types' lowest values inside and beside pieces that
    share a 16-byte unit (the row form);
  - generic regions whose x is their y, whose arrays overlap, and in a CUDA graph;
  - the row-pass ring of the 2-D stencil, on shapes that block windows would take.

Each case asks the rules on the host (plan_host) which form it runs."""
import numpy as np
import pytest

import oracle as O
import plan_host as P
from paper_2106_03219_gb300 import inputs
from paper_2106_03219_gb300 import omprt as R
from gpu_helpers import bits32, dev, host

pytestmark = pytest.mark.gpu

SCHEDS = {P.STATIC: R.SCHED_STATIC, P.CHUNKED: R.SCHED_STATIC_CHUNKED, P.DYNAMIC: R.SCHED_DYNAMIC,
          P.NONMONO: R.SCHED_NONMONOTONIC, P.GUIDED: R.SCHED_GUIDED}
ROWS = [(P.STATIC, 0, 3, 64), (P.CHUNKED, 201, 3, 64), (P.DYNAMIC, 61, 5, 128),
        (P.NONMONO, 203, 3, 96), (P.GUIDED, 33, 3, 64)]


def _res(dtype):
    import torch
    return torch.zeros(1, dtype=dtype, device="cuda")


def _same(a, b):
    """Bit-equal, or both NaN."""
    return np.array_equal(bits32(a)[~np.isnan(a)], bits32(b)[~np.isnan(b)]) and \
        np.array_equal(np.isnan(a), np.isnan(b))


@pytest.mark.parametrize("sched,chunk,G,T", ROWS)
def test_special_values_in_rows(rt, sched, chunk, G, T):
    """Every 7th element special, and NaN right beside the arrays: each result comes
    from its own operands."""
    import torch
    n = 200_003
    assert P.stream("axpy", n, sched, chunk, G, T)[0] == "rows"
    rng = np.random.default_rng(3)
    special = np.array([np.inf, -np.inf, np.nan, -0.0, 3e38, 1e-45], np.float32)
    xb, yb = inputs.f32_uniform01(n + 8, 0), inputs.f32_uniform01(n + 8, 1)
    for b in (xb, yb):
        at = rng.integers(0, n + 8, n // 7)
        b[at] = special[rng.integers(0, len(special), len(at))]
        b[:4] = b[4 + n:] = np.nan
    xd, yd = dev(xb), dev(yb)
    rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=xd[4:4 + n], y=yd[4:4 + n], alpha=3.0),
                     SCHEDS[sched], chunk, G, T)
    got = host(yd)
    with np.errstate(all="ignore"):
        assert _same(got[4:4 + n], O.axpy_f32(3.0, xb[4:4 + n], yb[4:4 + n]))
    assert _same(got[:4], yb[:4]) and _same(got[4 + n:], yb[4 + n:])
    # integers: the lowest value beside the array and inside it
    xi, yi = inputs.int32_uniform(n + 8, 2), inputs.int32_uniform(n + 8, 3)
    xi[:4] = xi[4 + n:] = yi[:4] = yi[4 + n:] = np.iinfo(np.int32).min
    yi[rng.integers(4, 4 + n, 999)] = np.iinfo(np.int32).min
    yd, r = dev(yi), _res(torch.int64)
    rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(xi)[4:4 + n], y=yd[4:4 + n], alpha=-7),
                     SCHEDS[sched], chunk, G, T, red=R.ReduceDesc(R.OP_SUM, 0, r.data_ptr()))
    want = O.axpy_i32(-7, xi[4:4 + n].copy(), yi[4:4 + n].copy())
    assert np.array_equal(host(yd)[4:4 + n], want)
    assert int(host(r)[0]) == O.sum_int(want)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("op", ["max", "min"])
@pytest.mark.parametrize("low", [False, True])
def test_extremes_in_rows(rt, op, low):
    """max / min of arrays of one value but for the type's end, whose neighbours
    outside the array are the other end; a NaN is skipped."""
    import torch
    n, G, T, chunk = 300_007, 3, 1024, 64
    assert P.stream("load_f32_max", n, P.DYNAMIC, chunk, G, T)[0] == "rows"
    end = np.float32(-np.inf if op == "max" else np.inf)
    a = np.full(n + 8, -end, np.float32)          # what must not leak in
    a[4:4 + n] = end if low else np.float32(1.5)
    if not low:
        a[[4, 1000, 3 + n]] = np.nan
        a[n // 2] = 2.5 if op == "max" else 0.5
    r = _res(torch.float64)
    rt.launch_region(R.loop_desc(R.BODY_NONE, n=n, x=dev(a)[4:4 + n], data_type=R.F32),
                     R.SCHED_DYNAMIC, chunk, G, T,
                     red=R.ReduceDesc(R.OP_MAX if op == "max" else R.OP_MIN, 0, r.data_ptr()))
    assert host(r)[0] == (end if low else 2.5 if op == "max" else 0.5)
    assert rt.sync_status() == 0


def _segments(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


@pytest.mark.parametrize("T", [64, 256])
def test_generic_x_is_y(rt, T):
    import torch
    seg = _segments([1000, 0, 3, 30_001, 9000, 8192])
    n, nseg = int(seg[-1]), len(seg) - 1
    assert P.tiles(n, nseg, 4, T) > 0
    x = inputs.f32_uniform01(n, 5)
    xd = dev(x)
    res = torch.full((3 * nseg,), -1.0, dtype=torch.float64, device="cuda")
    rt.launch_generic(dev(seg), R.loop_desc(R.BODY_DOT, n=n, x=xd, y=xd, alpha=1e-4), res, 4, T,
                      program=R.GENERIC_DOT_AXPY)
    got, new = host(res), host(xd)
    for s in range(nseg):
        xs = x[seg[s]:seg[s + 1]]
        exact = O.exact_dot_f32(xs, xs)
        assert abs(got[3 * s] - exact) <= 1e-6 * max(abs(exact), 1e-300), s
        want = O.axpy_f32(float(got[3 * s + 1]), xs, xs)
        assert np.array_equal(bits32(new[seg[s]:seg[s + 1]]), bits32(want)), s
    assert rt.sync_status() == 0


@pytest.mark.parametrize("shift", [1024, -1024])
def test_generic_overlapping_arrays(rt, shift):
    """y is x shifted by 1024 elements and no segment is longer: one team runs the
    segments in order, and each reads what the ones before it left."""
    import torch
    seg = _segments([1000, 1024, 0, 700, 1023, 512] * 5)
    n, nseg = int(seg[-1]), len(seg) - 1
    buf = inputs.f32_uniform01(n + 1024, 6)
    ox, oy = (0, shift) if shift > 0 else (-shift, 0)
    bd = dev(buf)
    res = torch.full((nseg,), -1.0, dtype=torch.float64, device="cuda")
    rt.launch_generic(dev(seg), R.loop_desc(R.BODY_AXPY, n=n, x=bd[ox:ox + n], y=bd[oy:oy + n],
                                            alpha=0.5), res, 1, 128)
    want = buf.copy()
    for s in range(nseg):
        a, b = seg[s], seg[s + 1]
        want[oy + a:oy + b] = O.axpy_f32(0.5, want[ox + a:ox + b].copy(), want[oy + a:oy + b].copy())
    assert np.array_equal(bits32(host(bd)), bits32(want))
    assert rt.sync_status() == 0


def test_generic_tiles_in_a_cuda_graph(rt):
    import torch
    seg = _segments([8191, 100, 30_000, 0, 24_577, 5])
    n, nseg = int(seg[-1]), len(seg) - 1
    assert P.tiles(n, nseg, 4, 256) > 0
    x, y = inputs.f32_uniform01(n, 7), inputs.f32_uniform01(n, 8)
    xd, yd, sd = dev(x), dev(y), dev(seg)
    res = torch.zeros(nseg, dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rt.launch_generic(sd, R.loop_desc(R.BODY_AXPY, n=n, x=xd, y=yd, alpha=0.25), res, 4, 256,
                          stream=s)
    want = O.axpy_f32(0.25, x, y)
    for _ in range(3):
        yd.copy_(dev(y))
        torch.cuda.synchronize()
        g.replay()
        assert np.array_equal(bits32(host(yd)), bits32(want))
        got = host(res)
        for k in range(nseg):
            exact = O.exact_sum_f32(want[seg[k]:seg[k + 1]])
            assert abs(got[k] - exact) <= 1e-6 * max(abs(exact), 1e-300), k
    assert rt.sync_status() == 0


@pytest.mark.parametrize("ny,nx,chunk,G,T", [(41, 4096, 64, 9, 256), (300, 1028, 128, 7, 96),
                                             (67, 2048, 33, 5, 480), (41, 4096, 5, 9, 256)])
def test_row_pass_ring_eager_and_in_a_graph(rt, ny, nx, chunk, G, T):
    """A budget too small for windows leaves static(c) with c in [4, 8) and [32, 128] to
    the ring; four 16 KB rows and more are opted in at the launch."""
    import torch
    assert not P.window(nx, ny, P.CHUNKED, chunk, G, T, budget=16)
    a = inputs.grid_f32(ny, nx, 7)
    ad = dev(a)
    want = bits32(O.stencil2d5(a))
    out = torch.full((ny, nx), -7.0, device="cuda")
    d = R.loop_desc(R.BODY_STENCIL2D5, n=ny * nx, x=ad, out=out, nx=nx, ny=ny)
    rt.set_stencil_stage_bytes(16)
    try:
        rt.launch_region(d, R.SCHED_STATIC_CHUNKED, chunk, G, T)
        assert np.array_equal(bits32(host(out)), want)
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            rt.launch_region(d, R.SCHED_STATIC_CHUNKED, chunk, G, T, stream=s)
    finally:
        rt.set_stencil_stage_bytes(226 * 1024)
    for _ in range(2):
        out.fill_(-7.0)
        torch.cuda.synchronize()
        g.replay()
        assert np.array_equal(bits32(host(out)), want)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("sched,chunk", [(P.STATIC, 0), (P.CHUNKED, 64), (P.DYNAMIC, 64),
                                         (P.NONMONO, 100)])
def test_block_windows_in_a_graph(rt, sched, chunk):
    import torch
    ny, nx, G, T = 41, 4096, 9, 256
    assert P.window(nx, ny, sched, chunk, G, T)
    a = inputs.grid_f32(ny, nx, 9)
    ad = dev(a)
    out = torch.full((ny, nx), -7.0, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rt.launch_region(R.loop_desc(R.BODY_STENCIL2D5, n=ny * nx, x=ad, out=out, nx=nx, ny=ny),
                         SCHEDS[sched], chunk, G, T, stream=s)
    for _ in range(2):
        out.fill_(-7.0)
        torch.cuda.synchronize()
        g.replay()
        assert np.array_equal(bits32(host(out)), bits32(O.stencil2d5(a)))
    assert rt.sync_status() == 0
