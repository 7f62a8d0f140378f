"""GPU: host threads launching the same kernel with different amounts of shared
memory, both beyond the 48 KB a kernel gets without its opt-in.

The opt-in is one value a kernel and device, shared by all host threads: while
each launch set it to its own size, a thread with a smaller launch could lower it
between another's opt-in and launch, and that launch was refused."""
import threading

import pytest

from paper_2106_03219_gb300 import omprt as R

pytestmark = pytest.mark.gpu

LAUNCHES = 4000


def _window(rt, k, torch):
    """2-D stencil, a team's block in shared memory: 12 or 3 teams of a 128 x 1024 grid."""
    x = torch.rand(128 * 1024, device="cuda")
    out = torch.empty_like(x)
    d = R.loop_desc(R.BODY_STENCIL2D5, n=x.numel(), x=x, out=out, nx=1024, ny=128)
    return (x, out), lambda st: rt.launch_region(d, R.SCHED_STATIC, 0, 12 if k else 3, 256, stream=st)


def _rows(rt, k, torch):
    """axpy under dynamic(64) in the row form: teams of 128 or 512 threads."""
    x = torch.rand(300_007, device="cuda")
    y = torch.rand_like(x)
    d = R.loop_desc(R.BODY_AXPY, n=x.numel(), x=x, y=y, alpha=0.0)
    return (x, y), lambda st: rt.launch_region(d, R.SCHED_DYNAMIC, 64, 5, 128 if k else 512,
                                               stream=st)


def _generic(rt, k, torch):
    """Generic regions through the tile ring: one team an SM, or several."""
    seg = torch.arange(0, 65 * 512, 512, device="cuda")
    x, y = torch.rand(64 * 512, device="cuda"), torch.rand(64 * 512, device="cuda")
    res = torch.zeros(64, dtype=torch.float64, device="cuda")
    d = R.loop_desc(R.BODY_DOT, n=x.numel(), x=x, y=y)
    teams = 3 * rt.sm_count if k else 8
    return (seg, x, y, res), lambda st: rt.launch_generic(seg, d, res, teams, 64, stream=st)


@pytest.mark.parametrize("make", [_window, _rows, _generic])
def test_two_threads_two_sizes(rt, make):
    import torch
    errors = []
    start = threading.Barrier(2)

    def work(k):
        own = R.Runtime(0)
        try:
            stream = torch.cuda.Stream()
            keep, launch = make(own, k, torch)
            torch.cuda.synchronize()
            start.wait()
            for _ in range(LAUNCHES):
                launch(stream)
            stream.synchronize()
            assert own.sync_status() == 0
            del keep
        except Exception as e:  # reported by the test's own thread
            errors.append(e)
        finally:
            torch.cuda.synchronize()
            own.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
