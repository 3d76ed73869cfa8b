"""The calls that a program built on the skeletons makes, as timed cases.

Each case is one pass through the Python API on device-resident data, with
the containers, plans and outputs that such a program keeps between calls
and the execution-plan table shipped with the package loaded once.  The
kinds are the library's workloads: the size sweep (Map, Reduce, Scan), the
dot product whose result the host reads, chains of 2D stencil steps, single
stencils with their adjoints, uneven batched instances, the differentiable
composed loss, the composed Map -> MapOverlap -> MapReduce call, and
MapArray.
"""
import os

import torch

import paper_1405_2915_gb300 as sk
from paper_1405_2915_gb300.autograd import composed_loss

_DEV = "cuda"
_W5 = (0.0, 0.125, 0.0, 0.125, 0.5, 0.125, 0.0, 0.125, 0.0)
_W9 = (0.0625, 0.125, 0.0625, 0.125, 0.25, 0.125, 0.0625, 0.125, 0.0625)
_STEPS = 10   # steps of a stencil chain

sk.skel_load_dispatch_table(os.path.join(os.path.dirname(os.path.abspath(sk.__file__)), "dispatch_gb300.tbl"))


def listed():
    return [
        # the bottom of the size sweep: short vectors in a latency-bound inner loop
        {"name": "sweep_1k", "kind": "sweep", "n": 1024},
        # one dot product of two 4 MiB vectors, read on the host (a solver's inner product)
        {"name": "dot_1m", "kind": "dot", "n": 1 << 20},
        # the middle of the sweep at a length that is no multiple of anything
        {"name": "sweep_5m", "kind": "sweep", "n": 5_000_011},
        # the top of the sweep: 1 GiB vectors
        {"name": "sweep_256m", "kind": "sweep", "n": 1 << 28},
        # ten chained smoothing steps, on a small grid that stays in L2 and on a large one
        {"name": "chain9_512", "kind": "chain", "fn": "stencil9", "boundary": "clamp", "rows": 512, "cols": 512},
        {"name": "chain5_8192", "kind": "chain", "fn": "stencil5", "boundary": "clamp", "rows": 8192, "cols": 8192},
        # one stencil and its adjoint on a grid with odd sides (rows at every alignment)
        {"name": "stencil9_4099", "kind": "stencil2d", "fn": "stencil9", "boundary": "clamp", "rows": 4097, "cols": 4099},
        # a 17-tap filter over a long signal, and its adjoint
        {"name": "stencil1d_64m", "kind": "stencil1d", "radius": 8, "boundary": "zero", "n": 1 << 26},
        # 4096 uneven instances in one captured plan
        {"name": "batched_4096", "kind": "batched", "instances": 4096, "lo": 64, "hi": 1 << 20, "plan": True},
        # loss and gradient of the composed pipeline (a training step on a grid)
        {"name": "loss_8192", "kind": "loss", "rows": 8192, "cols": 8192},
        # the composed call tanh -> 9-point stencil -> sum of squares, read on the host
        {"name": "compose_8192", "kind": "compose", "map": "tanh", "fn": "stencil9", "boundary": "clamp",
         "rows": 8192, "cols": 8192},
        # table lookups from a 4 MiB table, and a matrix-vector product by rows
        {"name": "maparray_16m", "kind": "maparray", "table": 1 << 20, "n": 1 << 24, "rows": 4096, "cols": 4096},
    ]


def _log(rng, lo, hi):
    return int(lo * (hi / lo) ** rng.random())


def _side(rng, lo, hi):
    s = _log(rng, lo, hi)
    return s if rng.random() < 0.5 else (s + 3) // 4 * 4   # half of them of any remainder


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "dot", "chain", "stencil2d", "stencil1d", "batched", "loss", "compose",
                       "maparray"])
    grid = {"rows": _side(rng, 256, 8192), "cols": _side(rng, 256, 8192)}
    boundary = rng.choice(["clamp", "clamp", "zero", "periodic"])
    if kind == "sweep":
        return {"kind": kind, "n": _log(rng, 1 << 10, 1 << 28)}
    if kind == "dot":
        return {"kind": kind, "n": _log(rng, 1 << 12, 1 << 26)}
    if kind in ("chain", "stencil2d"):
        return {"kind": kind, "fn": rng.choice(["stencil5", "stencil9"]), "boundary": boundary, **grid}
    if kind == "stencil1d":
        return {"kind": kind, "radius": rng.choice([1, 4, 8, 16]), "boundary": boundary,
                "n": _log(rng, 1 << 16, 1 << 26)}
    if kind == "batched":
        return {"kind": kind, "instances": _log(rng, 64, 4096), "lo": 64, "hi": _log(rng, 1 << 12, 1 << 20),
                "plan": rng.random() < 0.5}
    if kind == "loss":
        return {"kind": kind, **grid}
    if kind == "compose":
        return {"kind": kind, "map": rng.choice(["tanh", "tanh", "copy"]), "fn": rng.choice(["stencil5", "stencil9"]),
                "boundary": boundary, **grid}
    return {"kind": kind, "table": _log(rng, 1 << 12, 1 << 22), "n": _log(rng, 1 << 16, 1 << 24),
            "rows": _side(rng, 64, 8192), "cols": _side(rng, 64, 8192)}


# ------------------------------------------------------------------ inputs --
def _uniform(g, shape, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=g, device=_DEV, dtype=torch.float32).mul_(hi - lo).add_(lo)


def _lengths(case):
    """Instance lengths, log-uniform over [lo, hi]: one of each quantile."""
    b = case["instances"]
    q = (torch.arange(b, dtype=torch.float64) + 0.5) / b
    return (case["lo"] * (case["hi"] / case["lo"]) ** q).to(torch.int64)


def _inputs(case, seed):
    """The input tensors of a case, made from the seed."""
    g = torch.Generator(device=_DEV).manual_seed(seed)
    kind = case["kind"]
    if kind == "sweep":
        n = case["n"]
        xi = torch.randint(0, 101, (n,), generator=g, device=_DEV, dtype=torch.int32)
        return {"x": _uniform(g, n), "y": _uniform(g, n), "xi": xi}
    if kind == "dot":
        return {"x": _uniform(g, case["n"]), "y": _uniform(g, case["n"])}
    if kind == "stencil1d":
        return {"x": _uniform(g, case["n"]), "g": _uniform(g, case["n"])}
    if kind == "batched":
        order = torch.randperm(case["instances"], generator=torch.Generator().manual_seed(seed))
        offsets = torch.zeros(case["instances"] + 1, dtype=torch.int64)
        offsets[1:] = _lengths(case)[order].cumsum(0)
        return {"x": _uniform(g, int(offsets[-1])), "offsets": offsets.to(_DEV)}
    if kind == "maparray":
        return {"table": _uniform(g, case["table"]),
                "idx": torch.randint(0, case["table"], (case["n"],), generator=g, device=_DEV, dtype=torch.int32),
                "a": _uniform(g, case["cols"]), "m": _uniform(g, (case["rows"], case["cols"]))}
    shape = (case["rows"], case["cols"])
    if kind == "chain":
        return {"x": _uniform(g, shape, 0.0, 1.0)}
    if kind == "stencil2d":
        return {"x": _uniform(g, shape, 0.0, 1.0), "g": _uniform(g, shape)}
    return {"x": _uniform(g, shape)}


def prepare(case, seed):
    t = _inputs(case, seed)
    kind = case["kind"]
    s = {"case": case, "in": t}
    if kind == "loss":
        t["x"].requires_grad_(True)
        return s
    s["c"] = {k: sk.Container.from_tensor(v) for k, v in t.items()}
    out = {}
    if kind == "sweep":
        out = {"axpy": torch.empty_like(t["x"]), "sum": torch.empty(1, device=_DEV), "max": torch.empty(1, device=_DEV),
               "scan_i32": torch.empty_like(t["xi"]), "scan_f32": torch.empty_like(t["x"])}
    elif kind == "chain":
        out = {"y": torch.empty_like(t["x"]), "tmp": torch.empty_like(t["x"])}
    elif kind in ("stencil2d", "stencil1d"):
        out = {"y": torch.empty_like(t["x"]), "gx": torch.empty_like(t["x"])}
    elif kind == "batched":
        out = {"sumsq": torch.empty(case["instances"], device=_DEV), "scan": torch.empty_like(t["x"])}
    elif kind == "maparray":
        out = {"gather": torch.empty(case["n"], device=_DEV), "rowdot": torch.empty(case["rows"], device=_DEV)}
    s["out"] = out
    s["o"] = {k: sk.Container.from_tensor(v) for k, v in out.items()}
    if kind == "batched" and case["plan"]:
        s["plan"] = sk.Plan(s["c"]["x"], s["c"]["offsets"], s["o"]["sumsq"], s["o"]["scan"], True)
    return s


# -------------------------------------------------------------------- pass --
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "loss":
        x = s["in"]["x"]
        loss = composed_loss(x)
        (gx,) = torch.autograd.grad(loss, x)
        return [loss.detach(), gx]
    c, o, out = s["c"], s["o"], s["out"]
    if kind == "sweep":
        sk.skel_map("axpy", [c["x"], c["y"]], o["axpy"], [2.5])
        sk.skel_reduce("add", c["x"], o["sum"], host=False)
        sk.skel_reduce("max", c["x"], o["max"], host=False)
        sk.skel_scan("add", True, c["xi"], o["scan_i32"])
        sk.skel_scan("add", False, c["x"], o["scan_f32"])
        return [out["axpy"], out["sum"], out["max"], out["scan_i32"], out["scan_f32"]]
    if kind == "dot":
        return [sk.skel_mapreduce("mul", "add", [c["x"], c["y"]])]
    if kind == "chain":
        sk.skel_mapoverlap_chain(case["fn"], None, case["boundary"], _STEPS, c["x"], o["tmp"], o["y"])
        return [out["y"]]
    if kind == "stencil2d":
        sk.skel_mapoverlap(case["fn"], 1, None, case["boundary"], c["x"], o["y"])
        sk.skel_mapoverlap_bwd(case["fn"], 1, None, case["boundary"], c["g"], o["gx"])
        return [out["y"], out["gx"]]
    if kind == "stencil1d":
        sk.skel_mapoverlap("stencil1d", case["radius"], None, case["boundary"], c["x"], o["y"])
        sk.skel_mapoverlap_bwd("stencil1d", case["radius"], None, case["boundary"], c["g"], o["gx"])
        return [out["y"], out["gx"]]
    if kind == "batched":
        if case["plan"]:
            s["plan"].launch()
        else:
            sk.skel_batched(c["x"], c["offsets"], o["sumsq"], o["scan"], True)
        return [out["sumsq"], out["scan"]]
    if kind == "compose":
        return [sk.skel_compose_map_stencil_sumsq(case["map"], case["fn"], c["x"], boundary=case["boundary"])]
    sk.skel_maparray("gather", c["table"], c["idx"], o["gather"])
    sk.skel_maparray("rowdot", c["a"], c["m"], o["rowdot"])
    return [out["gather"], out["rowdot"]]


def work(case):
    kind = case["kind"]
    if kind == "sweep":     # axpy 12 B, two reductions 4 B each, two scans 8 B each
        return {"bytes": 36 * case["n"], "flops": 6 * case["n"]}
    if kind == "dot":
        return {"bytes": 8 * case["n"], "flops": 2 * case["n"]}
    if kind == "stencil1d":  # forward and adjoint, a read and a write each
        return {"bytes": 16 * case["n"], "flops": 4 * (2 * case["radius"] + 1) * case["n"]}
    if kind == "batched":   # values in, scan out, offsets, results
        n, b = int(_lengths(case).sum()), case["instances"]
        return {"bytes": 8 * n + 12 * b, "flops": 3 * n}
    if kind == "maparray":
        m = case["rows"] * case["cols"]
        return {"bytes": 8 * case["n"] + 4 * (case["table"] + m + case["rows"] + case["cols"]), "flops": 2 * m}
    n = case["rows"] * case["cols"]
    taps = 5 if case.get("fn") == "stencil5" else 9
    if kind == "chain":     # the grid in and out once
        return {"bytes": 8 * n, "flops": 2 * taps * _STEPS * n}
    if kind == "stencil2d":
        return {"bytes": 16 * n, "flops": 4 * taps * n}
    if kind == "compose":
        return {"bytes": 4 * n, "flops": (2 * taps + 2) * n}
    # loss: the forward reads x, the backward reads it again and writes the gradient
    return {"bytes": 12 * n, "flops": 50 * n}


# ------------------------------------------------------------------- exact --
def _pad2(x, boundary):
    """x with one ring of cells as the boundary reads them."""
    if boundary == "zero":
        return torch.nn.functional.pad(x, (1, 1, 1, 1))
    if boundary == "clamp":
        x = torch.cat([x[:1], x, x[-1:]], 0)
        return torch.cat([x[:, :1], x, x[:, -1:]], 1)
    x = torch.cat([x[-1:], x, x[:1]], 0)
    return torch.cat([x[:, -1:], x, x[:, :1]], 1)


def _stencil2(x, fn, boundary):
    w = _W5 if fn == "stencil5" else _W9
    rows, cols = x.shape
    p = _pad2(x, boundary)
    y = torch.zeros_like(x)
    for k, wk in enumerate(w):
        if wk:
            y.add_(p[k // 3:k // 3 + rows, k % 3:k % 3 + cols], alpha=wk)
    return y


def _stencil2_adjoint(g, fn, boundary):
    """The transposed stencil: every tap's weight goes back to the cell it read."""
    w = _W5 if fn == "stencil5" else _W9
    rows, cols = g.shape
    p = torch.zeros((rows + 2, cols + 2), dtype=g.dtype, device=g.device)
    for k, wk in enumerate(w):
        if wk:
            p[k // 3:k // 3 + rows, k % 3:k % 3 + cols].add_(g, alpha=wk)
    for _ in range(2):      # fold the ring's rows, then (transposed) its columns
        if boundary == "clamp":
            p[1].add_(p[0])
            p[-2].add_(p[-1])
        elif boundary == "periodic":
            p[-2].add_(p[0])
            p[1].add_(p[-1])
        p = p[1:-1].t()
    return p.contiguous()


def _weights1(r):
    w, c = [], 1.0
    for k in range(2 * r + 1):
        w.append(c / 4.0 ** r)
        c = c * (2 * r - k) / (k + 1)
    return torch.tensor(w, dtype=torch.float32).double().tolist()   # the library rounds them once


def _pad1(x, r, boundary):
    if boundary == "zero":
        return torch.nn.functional.pad(x, (r, r))
    if boundary == "clamp":
        return torch.cat([x[:1].expand(r), x, x[-1:].expand(r)])
    return torch.cat([x[-r:], x, x[:r]])


def exact(case, seed):
    t = {k: (v.double() if v.is_floating_point() else v) for k, v in _inputs(case, seed).items()}
    kind = case["kind"]
    x = t.get("x")
    if kind == "sweep":
        scan = x.cumsum(0)
        scan = torch.cat([scan.new_zeros(1), scan[:-1]])
        return [2.5 * x + t["y"], x.sum().reshape(1), x.max().reshape(1), None, scan]
    if kind == "dot":
        return [(x * t["y"]).sum().reshape(())]
    if kind == "chain":
        for _ in range(_STEPS):
            x = _stencil2(x, case["fn"], case["boundary"])
        return [x]
    if kind == "stencil2d":
        return [_stencil2(x, case["fn"], case["boundary"]), _stencil2_adjoint(t["g"], case["fn"], case["boundary"])]
    if kind == "stencil1d":
        r, n = case["radius"], case["n"]
        w = _weights1(r)
        p, q = _pad1(x, r, case["boundary"]), x.new_zeros(n + 2 * r)
        y = torch.zeros_like(x)
        for k, wk in enumerate(w):
            y.add_(p[k:k + n], alpha=wk)
            q[k:k + n].add_(t["g"], alpha=wk)
        gx = q[r:r + n].clone()
        if case["boundary"] == "clamp":
            gx[0] += q[:r].sum()
            gx[-1] += q[r + n:].sum()
        elif case["boundary"] == "periodic":
            gx[-r:] += q[:r]
            gx[:r] += q[r + n:]
        return [y, gx]
    if kind == "batched":
        lo, hi = t["offsets"][:-1], t["offsets"][1:]
        scan = torch.cat([x.new_zeros(1), x.cumsum(0)])
        sq = torch.cat([x.new_zeros(1), x.square().cumsum(0)])
        base = torch.repeat_interleave(scan[lo], hi - lo)
        return [sq[hi] - sq[lo], scan[1:] - base]
    if kind == "loss":
        n = x.numel()
        y = torch.tanh(x)
        u, s = _stencil2(y, "stencil9", "clamp"), y.cumsum(1)
        loss = u.square().sum() + s.square().sum() / n
        gs = 2.0 * s / n
        back = gs.sum(1, keepdim=True) - gs.cumsum(1) + gs     # the reverse scan of each row
        gx = (_stencil2_adjoint(2.0 * u, "stencil9", "clamp") + back) * (1.0 - y * y)
        return [loss.reshape(1), gx]
    if kind == "compose":
        y = torch.tanh(x) if case["map"] == "tanh" else x
        return [_stencil2(y, case["fn"], case["boundary"]).square().sum().reshape(())]
    return [t["table"][t["idx"].long()], t["m"] @ t["a"]]
