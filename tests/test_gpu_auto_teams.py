"""GPU parity: schedule(auto) launches with fewer vectors than threads, which
launch only the teams that get an iteration, and reductions of one team, which
finish without a ticket.  Sizes around whole teams of vectors, with and without
the vector path; integers and extrema exact, fp32 / bf16 sums within the bound."""
import numpy as np
import pytest

import oracle as O
from paper_2106_03219_gb300 import inputs
from paper_2106_03219_gb300 import omprt as R
from gpu_helpers import bits32, dev, fp_sum_ok, host

pytestmark = pytest.mark.gpu


def _res(f):
    import torch
    return torch.zeros(1, dtype=torch.float64 if f else torch.int64, device="cuda")


@pytest.mark.parametrize("T", [32, 512])
@pytest.mark.parametrize("off", [0, 1])
def test_short_reductions(rt, T, off):
    import torch
    for teams in (1, 2, 3):
        for vec in (4, 8, 16):
            for d in (-1, 0, 1):
                n = teams * T * vec + d
                a = inputs.int64_uniform(n + off, n)[off:]
                x = dev(np.concatenate([np.zeros(off, np.int64), a]))[off:]
                for op, want in ((R.OP_SUM, O.sum_int(a)), (R.OP_MIN, O.max_min(a, "min"))):
                    r, q = _res(False), _res(False)
                    rt.reduce(op, x, r, 0, 304, T)
                    R.reduce_noalloc(op, x, q, threads=T)
                    assert int(host(r)[0]) == want and int(host(q)[0]) == want, (n, op)
                f = -np.abs(inputs.f32_lognormal_signed(n + off, n)) - np.float32(1)
                xf = dev(f)[off:]
                r = _res(True)
                rt.reduce(R.OP_MAX, xf, r, 0, 304, T)
                assert host(r)[0] == O.max_min(f[off:], "max")
                for prec in (R.PREC_COMP_F64, R.PREC_COMP_F32):
                    rt.reduce(R.OP_SUM, xf, r, prec, 304, T)
                    assert fp_sum_ok(float(host(r)[0]), O.exact_sum_f32(f[off:]),
                                     O.exact_abs_sum_f32(f[off:]))[0], (n, prec)
    b = inputs.bf16_uniform_pm1(16 * T + 5, 1)
    xb = dev(b.view(np.int16)).view(torch.bfloat16)
    r = _res(True)
    rt.reduce(R.OP_SUM, xb, r, R.PREC_COMP_F64, 304, T)
    vals = (b.astype(np.uint32) << 16).view(np.float32)
    assert fp_sum_ok(float(host(r)[0]), O.exact_sum_bf16(b), O.exact_abs_sum_f32(vals))[0]
    assert rt.sync_status() == 0


@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 4097, 16391])
def test_short_auto_loops(rt, n):
    import torch
    for off in (0, 1):
        xb, yb = inputs.f32_uniform01(n + 8, 0), inputs.f32_uniform01(n + 8, 1)
        yd, r = dev(yb), _res(True)
        rt.launch_region(R.loop_desc(R.BODY_AXPY, n=n, x=dev(xb)[off:off + n],
                                     y=yd[off:off + n], alpha=3.0), R.SCHED_AUTO, 0, 600, 256,
                         red=R.ReduceDesc(R.OP_SUM, R.PREC_COMP_F64, r.data_ptr()))
        want = yb.copy()
        want[off:off + n] = O.axpy_f32(3.0, xb[off:off + n], yb[off:off + n])
        assert np.array_equal(bits32(host(yd)), bits32(want))
        exact = O.exact_sum_f32(want[off:off + n])
        assert fp_sum_ok(float(host(r)[0]), exact, exact)[0]
        out = torch.full((n + 8,), -7.0, device="cuda")
        xs = np.ascontiguousarray(xb[off:off + n])
        rt.launch_region(R.loop_desc(R.BODY_STENCIL1D3, n=n, x=dev(xb)[off:off + n],
                                     out=out[off:off + n]), R.SCHED_AUTO, 0, 600, 256)
        got = host(out)
        assert np.array_equal(bits32(got[off:off + n]), bits32(O.stencil1d3(xs)))
        assert (got[:off] == -7.0).all() and (got[off + n:] == -7.0).all()
    assert rt.sync_status() == 0
