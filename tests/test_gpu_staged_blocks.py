"""GPU parity: the staged form on team blocks that all start on 16 bytes and end in
a short chunk, at many chunk and team sizes, every schedule and reduction it has.

The rule that picks the form is asked on the host for each case, so that a
change of the rule cannot empty these tests unseen.  Maps and integer sums
bit-exact, fp32 and bf16 sums within the reduction bound."""
import numpy as np
import pytest

import oracle as O
import plan_host as P
from paper_2106_03219_gb300 import inputs
from paper_2106_03219_gb300 import omprt as R
from gpu_helpers import bits32, dev, fp_sum_ok, host

pytestmark = pytest.mark.gpu

SCHED = {P.DYNAMIC: R.SCHED_DYNAMIC, P.NONMONO: R.SCHED_NONMONOTONIC,
         P.CHUNKED: R.SCHED_STATIC_CHUNKED}


def _res(dtype):
    import torch
    return torch.zeros(1, dtype=dtype, device="cuda")


@pytest.mark.parametrize("sched", sorted(SCHED))
@pytest.mark.parametrize("chunk,T", [(256, 32), (64, 32), (64, 128), (128, 64), (68, 32)])
def test_axpy_short_last_chunks(rt, sched, chunk, T):
    for G in (1, 7, 64):
        for extra in (0, 4, chunk - 4):  # the last chunk of every block
            n = G * (70 * chunk + extra)
            assert P.stream("axpy", n, sched, chunk, G, T)[0] == "staged"
            x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
            yd = dev(y)
            rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(x), y=yd, alpha=3.0),
                             SCHED[sched], chunk, G, T)
            assert np.array_equal(bits32(host(yd)), bits32(O.axpy_f32(3.0, x, y))), (G, extra)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("tail", [1, 2, 3])
def test_array_end_inside_a_unit(rt, tail):
    """One team, or equal blocks but for the last: the array ends inside a unit."""
    for G, n in ((1, 64 * 70 + tail), (4, 4 * (64 * 70 + 4) - (4 - tail))):
        q, r = divmod(n, G)
        if any((g * q + min(g, r)) % 4 for g in range(G)):
            continue
        assert P.stream("axpy", n, P.DYNAMIC, 64, G, 64)[0] == "staged"
        x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
        yd = dev(y)
        rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(x), y=yd, alpha=3.0),
                         R.SCHED_DYNAMIC, 64, G, 64)
        assert np.array_equal(bits32(host(yd)), bits32(O.axpy_f32(3.0, x, y))), G
    assert rt.sync_status() == 0


@pytest.mark.parametrize("budget", [16, 2048, 16384, 32768, 65536, 131072])
def test_axpy_i32_budgets(rt, budget):
    import torch
    rt.set_stage_bytes(budget)
    staged = 0
    try:
        for chunk, T in ((64, 32), (256, 64), (256, 32), (64, 512)):
            n = 19 * (40 * chunk + 20)
            x, y = inputs.int32_uniform(n, 3), inputs.int32_uniform(n, 4)
            want = O.axpy_i32(3, x, y)
            staged += P.stream("axpy_i32_sum", n, P.DYNAMIC, chunk, 19, T, budget)[0] == "staged"
            yd, r = dev(y), _res(torch.int64)
            rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(x), y=yd, alpha=3),
                             R.SCHED_DYNAMIC, chunk, 19, T,
                             red=R.ReduceDesc(R.OP_SUM, 0, r.data_ptr()))
            assert np.array_equal(host(yd), want), (chunk, T)
            assert int(host(r)[0]) == O.sum_int(want), (chunk, T)
    finally:
        rt.set_stage_bytes(32768)
    assert staged >= (1 if budget >= 16384 else 0)
    assert rt.sync_status() == 0


@pytest.mark.parametrize("sched", sorted(SCHED))
@pytest.mark.parametrize("chunk,T", [(64, 32), (64, 64), (128, 32)])
def test_reductions(rt, sched, chunk, T):
    import torch
    G = 11
    n = G * (90 * chunk + 16)
    x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
    r = _res(torch.float64)
    kinds = set()

    def run(desc, op, prec, res, body):
        kinds.add((body, P.stream(body, n, sched, chunk, G, T)[0]))
        rt.launch_region(desc, SCHED[sched], chunk, G, T,
                         red=R.ReduceDesc(op, prec, res.data_ptr()))
        return host(res)[0]

    got = run(R.loop_desc(R.BODY_DOT, n=n, x=dev(x), y=dev(y)), R.OP_SUM, R.PREC_COMP_F64, r, "dot")
    exact = O.exact_dot_f32(x, y)
    assert fp_sum_ok(float(got), exact, exact)[0]
    a = inputs.f32_lognormal_signed(n, 2)
    got = run(R.loop_desc(R.BODY_NONE, n=n, x=dev(a), data_type=R.F32), R.OP_SUM, R.PREC_COMP_F64,
              r, "load_f32_sum")
    assert fp_sum_ok(float(got), O.exact_sum_f32(a), O.exact_abs_sum_f32(a))[0]
    got = run(R.loop_desc(R.BODY_NONE, n=n, x=dev(a), data_type=R.F32), R.OP_MAX, 0, r,
              "load_f32_max")
    assert got == O.max_min(a, "max")
    bits = inputs.bf16_uniform_pm1(n, 5)
    xb = dev(bits.view(np.int16)).view(torch.bfloat16)
    got = run(R.loop_desc(R.BODY_NONE, n=n, x=xb, data_type=R.BF16), R.OP_SUM, R.PREC_COMP_F64, r,
              "load_bf16_sum")
    vals = (bits.astype(np.uint32) << 16).view(np.float32)
    assert fp_sum_ok(float(got), O.exact_sum_bf16(bits), O.exact_abs_sum_f32(vals))[0]
    ri = _res(torch.int64)
    for a, body in ((inputs.int32_uniform(n, 3), "load_i32"), (inputs.int64_uniform(n, 4),
                                                               "load_i64")):
        dt = R.I32 if a.dtype == np.int32 else R.I64
        got = run(R.loop_desc(R.BODY_NONE, n=n, x=dev(a), data_type=dt), R.OP_SUM, 0, ri, body)
        assert int(got) == O.sum_int(a)
    assert {k for _, k in kinds} >= {"staged"}, kinds
    assert rt.sync_status() == 0


def test_staged_axpy_in_a_cuda_graph(rt):
    import torch
    n = 64 * (40 * 256 + 16)
    assert P.stream("axpy", n, P.DYNAMIC, 256, 64, 32)[0] == "staged"
    assert P.stream("axpy", n, P.CHUNKED, 64, 16, 128)[0] == "staged"
    x, y = inputs.f32_uniform01(n, 0), inputs.f32_uniform01(n, 1)
    xd, yd = dev(x), dev(y)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    d = R.loop_desc(R.BODY_AXPY, n=n, x=xd, y=yd, alpha=3.0)
    with torch.cuda.graph(g, stream=s):
        rt.launch_region(d, R.SCHED_DYNAMIC, 256, 64, 32, stream=s)
        rt.launch_region(d, R.SCHED_STATIC_CHUNKED, 64, 16, 128, stream=s)
    want = O.axpy_f32(3.0, x, O.axpy_f32(3.0, x, y))
    for _ in range(3):
        yd.copy_(dev(y))
        torch.cuda.synchronize()
        g.replay()
        assert np.array_equal(bits32(host(yd)), bits32(want))
    assert rt.sync_status() == 0
