"""GPU parity: the row form of static, static(c), dynamic(c), nonmonotonic
dynamic and guided (each lane's next row of its piece staged through shared memory).

Sizes put piece ends at every place of a 16-byte unit and of a row, blocks of
too few chunks beside long ones, teams of every buffer shape (two and more
stages of 128-byte rows, 64-byte rows, one stage), arrays 16 but not 128 bytes
aligned, and array ends inside a unit.  Maps and integer sums bit-exact, fp32
sums within the reduction bound; neighbours of the arrays untouched."""
import numpy as np
import pytest

import oracle as O
from paper_2106_03219_gb300 import inputs
from paper_2106_03219_gb300 import omprt as R
from gpu_helpers import bits32, dev, fp_sum_ok, host

pytestmark = pytest.mark.gpu

SCHEDS = [(R.SCHED_STATIC, 0), (R.SCHED_STATIC_CHUNKED, 32), (R.SCHED_STATIC_CHUNKED, 61),
          (R.SCHED_STATIC_CHUNKED, 1000), (R.SCHED_DYNAMIC, 64), (R.SCHED_DYNAMIC, 257),
          (R.SCHED_NONMONOTONIC, 96), (R.SCHED_GUIDED, 32), (R.SCHED_GUIDED, 301)]
SHAPES = [(1, 32), (3, 128), (5, 256), (2, 512), (3, 1024)]
NS = [40_961, 300_006, (1 << 20) + 3]


def _res(dtype):
    import torch
    return torch.zeros(1, dtype=dtype, device="cuda")


@pytest.mark.parametrize("sched,chunk", SCHEDS)
@pytest.mark.parametrize("G,T", SHAPES)
def test_axpy_rows_bit_exact(rt, sched, chunk, G, T):
    import torch
    for n in NS:
        for off in (0, 4):  # 16-byte offset: rows no longer start on a line
            xb, yb = inputs.f32_uniform01(n + 16, 0), inputs.f32_uniform01(n + 16, 1)
            xd, yd = dev(xb), dev(yb)
            rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=xd[off:off + n], y=yd[off:off + n],
                                         alpha=3.0), sched, chunk, G, T)
            want = yb.copy()
            want[off:off + n] = O.axpy_f32(3.0, xb[off:off + n], yb[off:off + n])
            assert np.array_equal(bits32(host(yd)), bits32(want)), (n, off)
        xi, yi = inputs.int32_uniform(n, 2), inputs.int32_uniform(n, 3)
        yd, r = dev(yi), _res(torch.int64)
        rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(xi), y=yd, alpha=-7), sched, chunk,
                         G, T, red=R.ReduceDesc(R.OP_SUM, 0, r.data_ptr()))
        want = O.axpy_i32(-7, xi, yi)
        assert np.array_equal(host(yd), want), n
        assert int(host(r)[0]) == O.sum_int(want), n
    assert rt.sync_status() == 0


@pytest.mark.parametrize("sched,chunk", [(R.SCHED_STATIC, 0), (R.SCHED_STATIC_CHUNKED, 61),
                                         (R.SCHED_DYNAMIC, 514), (R.SCHED_NONMONOTONIC, 96),
                                         (R.SCHED_GUIDED, 64)])
@pytest.mark.parametrize("G,T", SHAPES)
def test_value_reductions_rows(rt, sched, chunk, G, T):
    import torch
    n = 300_007
    run = lambda d, op, r: rt.launch_region(d, sched, chunk, G, T,
                                            red=R.ReduceDesc(op, R.PREC_COMP_F64, r.data_ptr()))
    f = _res(torch.float64)
    x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
    run(R.loop_desc(R.BODY_DOT, n=n, x=dev(x), y=dev(y)), R.OP_SUM, f)
    exact = O.exact_dot_f32(x, y)
    assert fp_sum_ok(float(host(f)[0]), exact, exact)[0]
    # every element negative (positive): a masked or padded one would show
    a = -np.abs(inputs.f32_lognormal_signed(n, 2)) - np.float32(1)
    run(R.loop_desc(R.BODY_NONE, n=n, x=dev(a), data_type=R.F32), R.OP_MAX, f)
    assert host(f)[0] == O.max_min(a, "max")
    run(R.loop_desc(R.BODY_NONE, n=n, x=dev(-a), data_type=R.F32), R.OP_MIN, f)
    assert host(f)[0] == O.max_min(-a, "min")
    run(R.loop_desc(R.BODY_NONE, n=n, x=dev(a), data_type=R.F32), R.OP_SUM, f)
    assert fp_sum_ok(float(host(f)[0]), O.exact_sum_f32(a), O.exact_abs_sum_f32(a))[0]
    bits = inputs.bf16_uniform_pm1(n, 5)
    xb = dev(bits.view(np.int16)).view(torch.bfloat16)
    run(R.loop_desc(R.BODY_NONE, n=n, x=xb, data_type=R.BF16), R.OP_SUM, f)
    vals = (bits.astype(np.uint32) << 16).view(np.float32)
    assert fp_sum_ok(float(host(f)[0]), O.exact_sum_bf16(bits), O.exact_abs_sum_f32(vals))[0]
    i = _res(torch.int64)
    for v in (inputs.int32_uniform(n, 3), inputs.int64_uniform(n, 4)):
        run(R.loop_desc(R.BODY_NONE, n=n, x=dev(v),
                        data_type=R.I32 if v.dtype == np.int32 else R.I64), R.OP_SUM, i)
        assert int(host(i)[0]) == O.sum_int(v)
    assert rt.sync_status() == 0


def test_rows_off_and_in_a_graph(rt):
    """Zero staging bytes: the plain form, same bytes; rows captured and replayed."""
    import torch
    n = 1_000_003
    x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
    once = O.axpy_f32(3.0, x, y)
    xd, yd = dev(x), dev(y)
    d = R.loop_desc(R.BODY_AXPY, n=n, x=xd, y=yd, alpha=3.0)
    rt.set_stage_bytes(0)
    try:
        rt.launch_region(d, R.SCHED_DYNAMIC, 256, 9, 128)
    finally:
        rt.set_stage_bytes(32768)
    assert np.array_equal(bits32(host(yd)), bits32(once))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rt.launch_region(d, R.SCHED_DYNAMIC, 256, 9, 128, stream=s)
        rt.launch_region(d, R.SCHED_STATIC, 0, 5, 256, stream=s)
    for _ in range(2):  # the dispatch counters are left at zero
        yd.copy_(dev(y))
        g.replay()
        want = O.axpy_f32(3.0, x, O.axpy_f32(3.0, x, y))
        assert np.array_equal(bits32(host(yd)), bits32(want))
    assert rt.sync_status() == 0
