"""The calls whose time matters to a user of this library, as cases that can be
prepared, run and checked one by one.

`listed()` gives the named cases, `draw(rng)` one more of the same ranges,
`prepare(case, seed)` what a program holds before the call (device arrays, loop
descriptors, a batch handle, model weights), `run(state)` one pass through the
public entry points, `work(case)` the bytes and operations of a pass, and
`exact(case, seed)` its floating results in 64 bits by plain torch.

A case's "path" names the entry points it goes through:
  loop      launch_region / launch_region_dist of a one-dimensional body under
            any schedule, and of the int32 axpy with its sum
  stencil2d launch_region of the 2-D 5-point stencil
  reduce    reduce, or reduce_noalloc
  batch     a batch handle's launch: many regions in one persistent kernel
  generic   launch_generic: sequential code with parallel regions, by segments
  mlp       mlp_loss_grad + mlp_adam (a training step), or mlp_forward
"""
import functools
import math

import torch

from paper_2106_03219_gb300 import inputs, learned
from paper_2106_03219_gb300 import omprt as R

ALPHA = 3.0
GENERIC_ALPHA = -1e-6   # contracts a segment's y a little each pass
C0, C1 = 0.5, 0.125     # loop_desc's stencil weights
LR, BETA1, BETA2, EPS = 1e-3, 0.9, 0.999, 1e-8
FIRST_STEP = 100        # the training step is one of a run under way

# schedule name -> (omprt schedule, chunk); dist is launch_region_dist with
# dist_schedule(static, T) and schedule(static, 1), the usual GPU composite
SCHEDULES = {
    "auto": (R.SCHED_AUTO, 0),
    "static": (R.SCHED_STATIC, 0),
    "static1": (R.SCHED_STATIC_CHUNKED, 1),
    "static8": (R.SCHED_STATIC_CHUNKED, 8),
    "static64": (R.SCHED_STATIC_CHUNKED, 64),
    "dynamic64": (R.SCHED_DYNAMIC, 64),
    "dynamic256": (R.SCHED_DYNAMIC, 256),
    "guided64": (R.SCHED_GUIDED, 64),
    "nonmonotonic256": (R.SCHED_NONMONOTONIC, 256),
    "learned": (R.SCHED_LEARNED, 0),
    "dist": (R.SCHED_STATIC_CHUNKED, 1),
}
OPS = {"sum": R.OP_SUM, "max": R.OP_MAX, "min": R.OP_MIN}
ELEM_BYTES = {"f32": 4, "bf16": 2, "i32": 4, "i64": 8}


def listed():
    """The named cases.  teams / threads 0 leave the choice to the runtime, as
    a program that does not tune its launches does."""
    return [
        # one small offloaded region with few teams: a loop inside a larger
        # host program, int32 data and a sum clause
        {"name": "region_i32_sum", "path": "loop", "body": "axpy_i32_sum", "schedule": "static",
         "n": 1 << 20, "teams": 4, "threads": 128},
        # the worksharing sweep's axpy under run-time dispatch
        {"name": "axpy_dynamic256", "path": "loop", "body": "axpy", "schedule": "dynamic256",
         "n": 1 << 26, "teams": 0, "threads": 0},
        # the default schedule on a length that no team count divides
        {"name": "axpy_static_ragged", "path": "loop", "body": "axpy", "schedule": "static",
         "n": 50_000_001, "teams": 1184, "threads": 256},
        # a short loop whose schedule the installed cost model picks
        {"name": "dot_learned", "path": "loop", "body": "dot", "schedule": "learned",
         "n": 1_000_003, "teams": 0, "threads": 0},
        # the worksharing sweep's grid under a chunked static schedule
        {"name": "stencil2d_static64", "path": "stencil2d", "schedule": "static64",
         "nx": 4096, "ny": 4096, "teams": 0, "threads": 0},
        # a grid whose rows are no whole vectors, mapping left to the runtime
        {"name": "stencil2d_odd_auto", "path": "stencil2d", "schedule": "auto",
         "nx": 3001, "ny": 2503, "teams": 0, "threads": 0},
        # the large reductions: fp32 with wide magnitudes, and bf16 of odd length
        {"name": "reduce_f32", "path": "reduce", "dtype": "f32", "op": "sum", "n": 1 << 28,
         "noalloc": False},
        {"name": "reduce_bf16_ragged", "path": "reduce", "dtype": "bf16", "op": "sum",
         "n": 100_000_003, "noalloc": False},
        # the smallest call: a reduction over a few pages of counters
        {"name": "reduce_i64_small", "path": "reduce", "dtype": "i64", "op": "sum", "n": 10_007,
         "noalloc": False},
        # thousands of short regions of uneven length in one launch
        {"name": "batch_4096", "path": "batch", "regions": 4096, "median": 10_000},
        # non-SPMD regions: two parallel loops a segment, sequential code between
        {"name": "generic_dot_axpy", "path": "generic", "program": "dot_axpy", "segments": 4096,
         "median": 8192},
        # a training step of the cost model at the batch the trainer uses
        {"name": "mlp_train", "path": "mlp", "train": True, "batch": 256},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _team_shape(rng):
    if rng.random() < 0.4:
        return {"teams": 0, "threads": 0}
    return {"teams": rng.randint(148, 1184), "threads": rng.choice((128, 256, 512, 1024))}


def draw(rng):
    """One more case of the listed ones' ranges."""
    path = rng.choice(("loop", "loop", "loop", "region", "stencil2d", "stencil2d", "reduce",
                       "reduce", "batch", "generic", "mlp"))
    if path == "loop":
        body = rng.choice(("axpy", "axpy", "dot", "stencil1d"))
        return {"path": "loop", "body": body, "schedule": rng.choice(sorted(SCHEDULES)),
                "n": _log_uniform(rng, 1 << 12, 1 << 26), **_team_shape(rng)}
    if path == "region":
        return {"path": "loop", "body": "axpy_i32_sum",
                "schedule": rng.choice(("static", "static1", "static8", "dynamic64")),
                "n": _log_uniform(rng, 1 << 14, 1 << 21), "teams": rng.randint(4, 64),
                "threads": rng.choice((128, 256, 512))}
    if path == "stencil2d":
        schedule = rng.choice(("auto", "static", "static1", "static8", "static64", "dynamic256"))
        nx, ny = _log_uniform(rng, 256, 4096), _log_uniform(rng, 256, 4096)
        if rng.random() < 0.5:
            nx -= nx % 32
        return {"path": "stencil2d", "schedule": schedule, "nx": nx, "ny": ny, **_team_shape(rng)}
    if path == "reduce":
        return {"path": "reduce", "dtype": rng.choice(("f32", "bf16", "i32", "i64")),
                "op": rng.choice(("sum", "sum", "max", "min")),
                "n": _log_uniform(rng, 1000, 1 << 27), "noalloc": rng.random() < 0.3}
    if path == "batch":
        return {"path": "batch", "regions": _log_uniform(rng, 64, 4096),
                "median": _log_uniform(rng, 1000, 10_000)}
    if path == "generic":
        return {"path": "generic", "program": rng.choice(("dot", "axpy", "dot_axpy")),
                "segments": _log_uniform(rng, 64, 4096), "median": _log_uniform(rng, 256, 8192)}
    return {"path": "mlp", "train": rng.random() < 0.7, "batch": _log_uniform(rng, 16, 2048)}


@functools.lru_cache(maxsize=None)
def _runtime():
    """The one context of a program, with the shipped cost model installed."""
    torch.cuda.init()
    rt = R.Runtime(torch.cuda.current_device())
    learned.Model.load().install(rt)
    return rt


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rand(n, gen):
    return torch.rand(n, generator=gen, device="cuda", dtype=torch.float32)


# -- sizes that follow from a case and its seed -------------------------------

def _trip_counts(case):
    """Lognormal trip counts of a batch's regions, their kinds and offsets: the
    case's, not the seed's."""
    n, kind, offset = inputs.batched_regions(case["regions"], median=float(case["median"]))
    return n.tolist(), kind.tolist(), offset.tolist()


def _segment_offsets(case):
    """Offsets of a generic region's uneven segments (the case's, not the seed's)."""
    g = inputs.rng(inputs.META_SEED)
    n = g.lognormal(math.log(case["median"]), 1.0, case["segments"]).clip(16, 1 << 17)
    return [0] + n.astype("int64").cumsum().tolist()


# -- inputs -------------------------------------------------------------------

def _loop_arrays(case, seed):
    g, n = _gen(seed), case["n"]
    if case["body"] == "axpy_i32_sum":
        lim = 1 << 20
        return tuple(torch.randint(-lim, lim, (n,), generator=g, device="cuda", dtype=torch.int32)
                     for _ in range(2))
    return _rand(n, g), _rand(n, g)


def _reduce_data(case, seed):
    g, n, dtype = _gen(seed), case["n"], case["dtype"]
    if dtype == "i32":
        return torch.randint(-(1 << 20), 1 << 20, (n,), generator=g, device="cuda",
                             dtype=torch.int32)
    if dtype == "i64":
        return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda",
                             dtype=torch.int64)
    if dtype == "bf16":
        return _rand(n, g).mul_(2).sub_(1).to(torch.bfloat16)
    x = torch.randn(n, generator=g, device="cuda").mul_(3.0).exp_()   # lognormal, sigma 3
    return x.mul_(_rand(n, g).sub_(0.5).sign_())                      # with random signs


def _batch_arrays(case, seed):
    n, kind, offset = _trip_counts(case)
    total = offset[-1] + (n[-1] + 63) // 64 * 64
    g = _gen(seed)
    return n, kind, offset, _rand(total, g), _rand(total, g)


def _generic_arrays(case, seed):
    seg = _segment_offsets(case)
    g = _gen(seed)
    return seg, _rand(seg[-1], g), _rand(seg[-1], g)


def _mlp_arrays(case, seed):
    g, B = _gen(seed), case["batch"]
    randn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    parts = []
    for fan_in, fan_out in ((16, 64), (64, 64), (64, 12)):
        parts += [randn(fan_out * fan_in) * math.sqrt(2.0 / fan_in), randn(fan_out) * 0.05]
    params = torch.cat(parts)
    x, target = randn(B, 16), randn(B, 12)
    # moments of a run under way
    m, v = randn(params.numel()) * 1e-2, randn(params.numel()).square() * 1e-3 + 1e-4
    return params, x, target, m, v


class _BatchHandle:
    """Destroys the batch with the state that holds it."""

    def __init__(self, batch):
        self.batch = batch

    def __del__(self):
        self.batch.destroy()


def prepare(case, seed):
    """What a program holds before the call."""
    rt, path = _runtime(), case["path"]
    s = {"case": case, "rt": rt}
    if path == "loop":
        body, n = case["body"], case["n"]
        x, y = _loop_arrays(case, seed)
        s["red"], s["out"] = None, {}
        if body == "stencil1d":
            s["desc"] = R.loop_desc(R.BODY_STENCIL1D3, n=n, x=x, out=y, c0=C0, c1=C1)
            s["out"]["out"] = y
        elif body == "dot":
            s["desc"] = R.loop_desc(R.BODY_DOT, n=n, x=x, y=y)
        else:
            s["desc"] = R.loop_desc(R.BODY_AXPY, n=n, x=x, y=y, alpha=ALPHA)
            s["out"]["y"] = y
        if body in ("dot", "axpy_i32_sum"):
            result = torch.zeros(1, device="cuda",
                                 dtype=torch.float64 if body == "dot" else torch.int64)
            s["red"] = R.ReduceDesc(R.OP_SUM, R.PREC_COMP_F64, result.data_ptr())
            s["out"]["sum"] = result
    elif path == "stencil2d":
        nx, ny = case["nx"], case["ny"]
        x = _rand(nx * ny, _gen(seed))
        out = torch.empty_like(x)
        s["red"], s["out"] = None, {"out": out}
        s["desc"] = R.loop_desc(R.BODY_STENCIL2D5, n=nx * ny, x=x, out=out, nx=nx, ny=ny, c0=C0,
                                c1=C1)
    elif path == "reduce":
        s["data"] = _reduce_data(case, seed)
        s["result"] = torch.zeros(1, device="cuda", dtype=torch.int64 if case["dtype"][0] == "i"
                                  else torch.float64)
    elif path == "batch":
        n, kind, offset, x, y = _batch_arrays(case, seed)
        out = torch.zeros_like(x)
        res = torch.zeros(len(n), dtype=torch.float64, device="cuda")
        descs, reds = [], []
        for r, (m, k, o) in enumerate(zip(n, kind, offset)):
            red = None
            if k == inputs.KIND_AXPY:
                descs.append(R.loop_desc(R.BODY_AXPY, n=m, x=x[o:], y=y[o:], alpha=ALPHA))
            elif k == inputs.KIND_DOT:
                descs.append(R.loop_desc(R.BODY_DOT, n=m, x=x[o:], y=y[o:]))
                red = res.data_ptr() + 8 * r
            else:
                descs.append(R.loop_desc(R.BODY_STENCIL1D3, n=m, x=x[o:], out=out[o:], c0=C0,
                                         c1=C1))
            reds.append(R.ReduceDesc(R.OP_SUM, R.PREC_COMP_F64, red))
        s["handle"] = _BatchHandle(rt.batch_create(descs, reds, 32768))
        s["keep"] = (x,)
        s["out"] = {"y": y, "out": out, "res": res}
    elif path == "generic":
        seg, x, y = _generic_arrays(case, seed)
        both = case["program"] == "dot_axpy"
        s["program"] = R.GENERIC_DOT_AXPY if both else R.GENERIC_REDUCE
        s["seg"] = torch.tensor(seg, dtype=torch.int64, device="cuda")
        s["result"] = torch.zeros((3 if both else 1) * (len(seg) - 1), dtype=torch.float64,
                                  device="cuda")
        s["desc"] = R.loop_desc(R.BODY_AXPY if case["program"] == "axpy" else R.BODY_DOT,
                                n=seg[-1], x=x, y=y, alpha=GENERIC_ALPHA)
        s["out"] = {"result": s["result"]}
        if case["program"] != "dot":
            s["out"]["y"] = y
    else:
        params, x, target, m, v = _mlp_arrays(case, seed)
        if case["train"]:
            s.update(params=params, x=x, target=target, m=m, v=v, grad=torch.zeros_like(params),
                     loss=torch.zeros(1, device="cuda"), step=FIRST_STEP)
        else:
            s.update(params=params, x=x, y=torch.zeros(case["batch"], 12, device="cuda"))
    return s


def run(s):
    """One pass through the public entry points."""
    case, rt = s["case"], s["rt"]
    path = case["path"]
    if path in ("loop", "stencil2d"):
        sched, chunk = SCHEDULES[case["schedule"]]
        if case["schedule"] == "dist":
            threads = case["threads"] or 256
            rt.launch_region_dist(s["desc"], threads, sched, chunk, case["teams"], threads,
                                  red=s["red"])
        else:
            rt.launch_region(s["desc"], sched, chunk, case["teams"], case["threads"],
                             red=s["red"])
        return s["out"]
    if path == "reduce":
        (R.reduce_noalloc if case["noalloc"] else rt.reduce)(OPS[case["op"]], s["data"],
                                                             s["result"])
        return s["result"]
    if path == "batch":
        s["handle"].batch.launch()
        return s["out"]
    if path == "generic":
        rt.launch_generic(s["seg"], s["desc"], s["result"], program=s["program"])
        return s["out"]
    if not case["train"]:
        rt.mlp_forward(s["params"], s["x"], s["y"])
        return s["y"]
    rt.mlp_loss_grad(s["params"], s["x"], s["target"], s["grad"], s["loss"])
    rt.mlp_adam(s["params"], s["grad"], s["m"], s["v"], s["step"], lr=LR, beta1=BETA1,
                beta2=BETA2, eps=EPS)
    s["step"] += 1
    return {k: s[k] for k in ("grad", "loss", "params", "m", "v")}


def work(case):
    """Bytes (each input read once, each output written once) and operations."""
    path = case["path"]
    if path == "loop":
        b, f = {"axpy": (12, 2), "axpy_i32_sum": (12, 3), "dot": (8, 2),
                "stencil1d": (8, 4)}[case["body"]]
        return {"bytes": b * case["n"], "flops": f * case["n"]}
    if path == "stencil2d":
        n = case["nx"] * case["ny"]
        return {"bytes": 8 * n, "flops": 6 * n}
    if path == "reduce":
        return {"bytes": ELEM_BYTES[case["dtype"]] * case["n"], "flops": case["n"]}
    if path == "batch":
        n, kind, _ = _trip_counts(case)
        return {"bytes": sum((8, 12)[k == inputs.KIND_AXPY] * m for m, k in zip(n, kind)),
                "flops": sum((2, 4)[k == inputs.KIND_STENCIL1D] * m for m, k in zip(n, kind))}
    if path == "generic":
        n = _segment_offsets(case)[-1]
        b, f = {"dot": (8, 2), "axpy": (12, 3), "dot_axpy": (12, 5)}[case["program"]]
        return {"bytes": b * n, "flops": f * n}
    B, P = case["batch"], R.MLP_NPARAM
    if not case["train"]:
        return {"bytes": 4 * (P + 28 * B), "flops": 2 * P * B}
    return {"bytes": 4 * (8 * P + 28 * B), "flops": 6 * P * B + 15 * P}


# -- 64-bit results by plain torch ----------------------------------------------

def _exact_stencil1d(x):
    x = x.double()
    out = x.clone()
    out[1:-1] = C0 * x[1:-1] + C1 * (x[:-2] + x[2:])
    return out


def _exact_mlp(case, seed):
    params, x, target, m, v = _mlp_arrays(case, seed)
    p = params.double().requires_grad_(case["train"])
    w1, b1, w2, b2, w3, b3 = p.split([1024, 64, 4096, 64, 768, 12])
    h = torch.relu(x.double() @ w1.view(64, 16).T + b1)
    h = torch.relu(h @ w2.view(64, 64).T + b2)
    y = h @ w3.view(12, 64).T + b3
    if not case["train"]:
        return y
    loss = (y - target.double()).square().mean()
    (g,) = torch.autograd.grad(loss, p)
    # the call takes its hyperparameters in fp32
    lr, b1_, b2_, eps = (float(torch.tensor(h, dtype=torch.float32)) for h in
                         (LR, BETA1, BETA2, EPS))
    m = b1_ * m.double() + (1 - b1_) * g
    v = b2_ * v.double() + (1 - b2_) * g * g
    step = lr * (m / (1 - b1_ ** FIRST_STEP)) / ((v / (1 - b2_ ** FIRST_STEP)).sqrt() + eps)
    return {"grad": g, "loss": loss.detach().reshape(1), "params": p.detach() - step, "m": m,
            "v": v}


def exact(case, seed):
    """The floating results of run() in 64 bits, laid out the same."""
    path = case["path"]
    if path == "loop":
        x, y = _loop_arrays(case, seed)
        if case["body"] == "axpy":
            return {"y": y.double().add_(x.double(), alpha=ALPHA)}
        if case["body"] == "dot":
            return {"sum": (x.double() * y.double()).sum().reshape(1)}
        if case["body"] == "stencil1d":
            return {"out": _exact_stencil1d(x)}
        return None
    if path == "stencil2d":
        x = _rand(case["nx"] * case["ny"], _gen(seed)).double().view(case["ny"], case["nx"])
        out = x.clone()
        out[1:-1, 1:-1] = C0 * x[1:-1, 1:-1] + C1 * (x[:-2, 1:-1] + x[2:, 1:-1] +
                                                     x[1:-1, :-2] + x[1:-1, 2:])
        return {"out": out.view(-1)}
    if path == "reduce":
        if case["dtype"][0] == "i":
            return None
        x = _reduce_data(case, seed).double()
        return {"sum": x.sum, "max": x.max, "min": x.min}[case["op"]]().reshape(1)
    if path == "batch":
        n, kind, offset, x, y = _batch_arrays(case, seed)
        yy, out = y.double(), torch.zeros_like(x, dtype=torch.float64)
        res = torch.zeros(len(n), dtype=torch.float64, device="cuda")
        for r, (m, k, o) in enumerate(zip(n, kind, offset)):
            xs, ys = x[o:o + m].double(), yy[o:o + m]
            if k == inputs.KIND_AXPY:
                ys.add_(xs, alpha=ALPHA)
            elif k == inputs.KIND_DOT:
                res[r] = (xs * ys).sum()
            else:
                out[o:o + m] = _exact_stencil1d(xs)
        return {"y": yy, "out": out, "res": res}
    if path == "generic":
        seg, x, y = _generic_arrays(case, seed)
        x, y = x.double(), y.double()
        off = torch.tensor(seg, device="cuda")
        which = torch.repeat_interleave(torch.arange(len(seg) - 1, device="cuda"), off.diff())
        total = lambda t: torch.zeros(len(seg) - 1, dtype=torch.float64,
                                      device="cuda").index_add_(0, which, t)
        if case["program"] == "dot":
            return {"result": total(x * y)}
        if case["program"] == "axpy":
            y = y + GENERIC_ALPHA * x
            return {"result": total(y), "y": y}
        v = total(x * y)
        a = v * GENERIC_ALPHA
        y = y + a[which] * x
        return {"result": torch.stack((v, a, total(y)), 1).view(-1), "y": y}
    return _exact_mlp(case, seed)
