"""The work whose speed this library is kept to: what its users have it do, as cases.

A case is a dict of plain values. listed() gives the fixed ones, draw() more of the same ranges; prepare() makes what
a program holds before the call (launches, an analysed graph, a captured batch), run() is one pass through the public
entry points, work() what the pass cannot do without, exact() its results from numpy alone where they have a closed
form. The kinds:

  call     one small graph from pinned host arrays to its finished state: ingest, analysis, one execution, status
  analyze  ingest and analysis of a launch stream, the DAG left as CSR in device memory
  execute  one execution of an analysed graph
  replay   an analysed graph executed several times in one launch (no analysis)
  stitch   the same, each replay joined to the next by the edges between two copies of the trace
  capture  many independent graphs analysed as one batch and executed once
  batch    a captured batch executed again, every graph several times

Every result is an integer. Bodies are SPIN (and FMA, for the float loop) with a few iterations, so that runtime
overhead is what a pass costs; the iteration count comes from the seed, within a narrow range, as do the traces.
"""
import math

import numpy as np
import torch

from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

RING, OWNED = grt.RT_EXEC_RING, grt.RT_EXEC_OWNED


def listed():
    return [
        # the smallest call, where latency and launches count: the 1-D stencil of 1600 launches, from the host
        dict(name="call_stencil_1d", kind="call", pieces=16, steps=100, cells=1024),
        # the same small graph captured and replayed, as a time loop replays its trace
        dict(name="replay_stencil_1d", kind="replay", trace="stencil_1d", pieces=16, steps=100, cells=1024,
             replays=4, body="COUNTER"),
        # one request of the served stream analysed alone: an odd size, rectangles of every shape, default tile
        dict(name="analyze_request", kind="analyze", trace="rects", n=5317, grid=1024, side0=4, side1=256,
             tile_w=0, tile_h=0, source="host", bounds=32),
        # the Task Bench grid of the benchmark, at the tile its tuner picks, launches already on the device
        dict(name="analyze_taskbench", kind="analyze", trace="taskbench", pattern="random", width=1024, steps=1000,
             encode="region", tile_w=32, tile_h=4, source="device", bounds=64),
        # explicit dependences (no rectangles), ragged width, from the host
        dict(name="analyze_explicit", kind="analyze", trace="taskbench", pattern="random", width=777, steps=431,
             encode="explicit", tile_w=0, tile_h=0, source="host", bounds=64),
        # the large analysis: a million launches of 1-4 rectangles on 4096 x 4096
        dict(name="analyze_rects_1m", kind="analyze", trace="rects", n=1000000, grid=4096, side0=16, side1=1024,
             tile_w=16, tile_h=32, source="device", bounds=64),
        # a wide wavefront graph under the policy and shape the tuner picks for it
        dict(name="execute_stencil_tuned", kind="execute", trace="taskbench", pattern="stencil", width=1024,
             steps=1000, body="SPIN", iters=8, policy="owned", blocks=32, warps=1, claim=1, keep=16),
        # an irregular one as a program that tunes nothing runs it
        dict(name="execute_random_default", kind="execute", trace="taskbench", pattern="random", width=1024,
             steps=300, body="SPIN", iters=8, policy="ring", blocks=0, warps=0, claim=0, keep=0),
        # a narrow, deep graph of floating-point tasks of about half a microsecond, one ready task per claim: the
        # granularity a runtime's overhead is measured at
        dict(name="execute_fma_narrow", kind="execute", trace="taskbench", pattern="stencil", width=32, steps=1000,
             body="FMA", iters=256, policy="ring", blocks=0, warps=0, claim=1, keep=0),
        # a short trace replayed with no barrier between its replays
        dict(name="stitch_stencil", kind="stitch", pattern="stencil", width=1024, steps=100, replays=20, iters=8),
        # requests that waited together, analysed as one batch and executed
        dict(name="capture_requests", kind="capture", graphs=43, n_lo=32, n_hi=16384, side0=4, side1=256, grid=1024,
             tile_w=16, tile_h=32),
        # the batched form: independent graphs of mixed size and pattern, each replayed
        dict(name="batch_replay", kind="batch", graphs=640, n_lo=64, n_hi=65536, replays=20, tile_w=8, tile_h=8,
             iters=8, blocks=304, warps=8, claim=16, keep=32),
    ]


def _log(rng, a, b):
    return int(min(max(math.floor(math.exp(rng.uniform(math.log(a), math.log(b + 1)))), a), b))


def draw(rng):
    kind = rng.choice(["call", "analyze", "analyze", "analyze", "execute", "execute", "replay", "stitch", "capture",
                       "batch"])
    if kind == "call":
        return dict(kind=kind, pieces=_log(rng, 3, 96), steps=_log(rng, 5, 400), cells=_log(rng, 16, 2048))
    if kind == "analyze":
        source, bounds = rng.choice(["host", "device"]), rng.choice([32, 64])
        if rng.random() < 0.5:
            tile = rng.choice([(0, 0), (16, 32), (16, 16), (32, 16), (8, 32)])
            grid = rng.choice([1024, 2048, 4096])
            return dict(kind=kind, trace="rects", n=_log(rng, 32, 100000), grid=grid, side0=4, side1=grid // 4,
                        tile_w=tile[0], tile_h=tile[1], source=source, bounds=bounds)
        tile = rng.choice([(0, 0), (8, 8), (16, 8), (32, 4)])
        encode = rng.choice(["region", "region", "explicit"])
        # random fan-in: the other patterns' graphs are the same for every seed
        return dict(kind=kind, trace="taskbench", pattern="random", width=_log(rng, 8, 1024), steps=_log(rng, 8, 1000),
                    encode=encode, tile_w=tile[0], tile_h=tile[1], source=source, bounds=bounds)
    if kind == "execute":
        pattern = rng.choice(["stencil", "butterfly", "random"])
        width = 1 << rng.randint(3, 10) if pattern == "butterfly" else _log(rng, 8, 1024)
        shape = rng.choice([("owned", 32, 1, 1, 16), ("owned", 64, 1, 2, 16), ("ring", 0, 0, 0, 0),
                            ("ring", 0, 0, 0, 0), ("ring", 152, 4, 4, 8), ("ring", 0, 0, 1, 0)])
        body, iters = rng.choice([("SPIN", 8), ("SPIN", _log(rng, 8, 512)), ("FMA", _log(rng, 16, 1024))])
        return dict(kind=kind, trace="taskbench", pattern=pattern, width=width, steps=_log(rng, 20, 1000), body=body,
                    iters=iters, policy=shape[0], blocks=shape[1], warps=shape[2], claim=shape[3], keep=shape[4])
    if kind == "replay":
        if rng.random() < 0.5:
            return dict(kind=kind, trace="stencil_1d", pieces=_log(rng, 3, 96), steps=_log(rng, 5, 400),
                        cells=_log(rng, 16, 2048), replays=rng.randint(2, 8), body="COUNTER")
        return dict(kind=kind, trace="taskbench", pattern=rng.choice(["stencil", "random"]), width=_log(rng, 8, 1024),
                    steps=_log(rng, 10, 100), replays=rng.randint(2, 20), body="SPIN", iters=_log(rng, 8, 256))
    if kind == "stitch":
        return dict(kind=kind, pattern=rng.choice(["stencil", "random"]), width=_log(rng, 8, 1024),
                    steps=_log(rng, 10, 100), replays=rng.randint(2, 20), iters=_log(rng, 8, 64))
    if kind == "capture":
        return dict(kind=kind, graphs=_log(rng, 2, 64), n_lo=32, n_hi=_log(rng, 256, 16384), side0=4, side1=256,
                    grid=1024, tile_w=16, tile_h=32)
    return dict(kind=kind, graphs=_log(rng, 8, 640), n_lo=64, n_hi=_log(rng, 1024, 65536), replays=rng.randint(1, 20),
                tile_w=8, tile_h=8, iters=_log(rng, 8, 64), blocks=0, warps=0, claim=0, keep=0)


# ----------------------------------------------------------------------------------------------------------------
def _iters(case, seed):
    """Body iterations: the case's, plus 0..7 from the seed."""
    return int(case["iters"]) + int(seed) % 8


def _requests(case, seed):
    """Graphs of random rectangles, task counts log-uniform, each on its own grid (requests share no data). The case
    alone gives the task counts, the seed the rectangles."""
    rng = np.random.Generator(np.random.PCG64(case["graphs"]))
    sizes = tg.loguniform_int(rng, case["n_lo"], case["n_hi"], case["graphs"])
    return [tg.random_rects(grid=(case["grid"], case["grid"]), n=int(m), side=(case["side0"], case["side1"]),
                            seed=seed * 1009 + k) for k, m in enumerate(sizes)]


def _batch_specs(case, seed):
    """(width, steps, pattern, seed) of a batch's graphs: the case gives their sizes and patterns, the seed the rest."""
    specs = tg.batch_graph_specs(case["graphs"], (case["n_lo"], case["n_hi"]), seed=case["graphs"])
    return [(w, t, pattern, seed * 100003 + k) for k, (w, t, pattern, _) in enumerate(specs)]


def _trace(case, seed):
    if case["trace"] == "stencil_1d":
        return tg.stencil_1d(case["pieces"], case["steps"], case["cells"])
    if case["trace"] == "rects":
        return tg.random_rects(grid=(case["grid"], case["grid"]), n=case["n"], side=(case["side0"], case["side1"]),
                               seed=seed)
    return tg.taskbench(case["width"], case["steps"], case["pattern"], seed=seed, encode=case.get("encode", "region"))


def _arrays(tr, source, bounds=64):
    """(req_off, lo, hi, priv, pred_off, pred, body_arg) in pinned host or device memory; 32- or 64-bit bounds."""
    lo, hi = (a.astype(np.int32 if bounds == 32 else np.int64) for a in (tr.lo, tr.hi))
    arrs = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)) for a in
            (tr.req_off, lo, hi, tr.priv, tr.pred_off, tr.pred, tr.body_arg)]
    return [None if a is None else (a.cuda() if source == "device" else a.pin_memory()) for a in arrs]


def _counters(case, seed):
    """Starting values of the pieces' counters."""
    g = np.random.Generator(np.random.PCG64(seed))
    return torch.from_numpy(g.integers(-1 << 31, 1 << 31, size=case["pieces"], dtype=np.int64).astype(np.int32)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "call":
        tr = tg.stencil_1d(case["pieces"], case["steps"], case["cells"])
        s["start"] = _counters(case, seed)
        s["state"] = torch.empty_like(s["start"])
        s["graph"] = grt.Graph(1, tr.dom_lo, tr.dom_hi, body=grt.RT_BODY_COUNTER, state=s["state"])
        s["launches"] = _arrays(tr, "host")
    elif kind == "analyze":
        tr = _trace(case, seed)
        s["graph"] = grt.Graph(2, tr.dom_lo, tr.dom_hi, tile=(case["tile_w"], case["tile_h"]))
        s["launches"] = _arrays(tr, case["source"], case["bounds"])
        s["csr"] = _csr_buffers(tr.n, 48 * tr.n if case["trace"] == "rects" else
                                _grid_edges("random", case["width"], case["steps"]))
    elif kind in ("execute", "replay"):
        tr = _trace(case, seed)
        if case["body"] == "COUNTER":
            s["start"] = _counters(case, seed)
            s["state"] = torch.empty_like(s["start"])
            g = grt.Graph(1, tr.dom_lo, tr.dom_hi, body=grt.RT_BODY_COUNTER, state=s["state"])
        else:
            s["out"] = torch.zeros(tr.n, dtype=torch.int32, device="cuda")
            body = grt.RT_BODY_FMA if case["body"] == "FMA" else grt.RT_BODY_SPIN
            g = grt.Graph(2, tr.dom_lo, tr.dom_hi, body=body, spin_iters=_iters(case, seed), out=s["out"])
        g.launch(*_arrays(tr, "device"))
        g.analyze()
        if kind == "execute":
            g.exec_policy(OWNED if case["policy"] == "owned" else RING)
            g.exec_config(case["blocks"], case["warps"], case["claim"], case["keep"])
        s["graph"] = g
    elif kind == "stitch":
        tr = tg.taskbench(case["width"], case["steps"], case["pattern"], seed=seed)
        s["out"] = torch.zeros(case["replays"] * tr.n, dtype=torch.int32, device="cuda")
        g = grt.Graph(2, tr.dom_lo, tr.dom_hi, body=grt.RT_BODY_SPIN, spin_iters=_iters(case, seed), out=s["out"])
        g.launch(*_arrays(tg.concat([tr, tr]), "device"))
        g.analyze()
        s["graph"] = g
    elif kind == "capture":
        s["traces"] = _requests(case, seed)
        n = sum(t.n for t in s["traces"])
        s["out"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["csr"] = _csr_buffers(n, 48 * n)
        s["inputs"] = [torch.from_numpy(a).cuda() for a in grt.concat_inputs(s["traces"])]
        s["iters"] = 8 + int(seed) % 8
    else:
        traces = [tg.batch_graph(sp) for sp in _batch_specs(case, seed)]
        s["out"] = torch.zeros(sum(t.n for t in traces), dtype=torch.int32, device="cuda")
        inputs = [torch.from_numpy(a).cuda() for a in grt.concat_inputs(traces)]
        s["batch"] = grt.Batch.capture(traces, body=grt.RT_BODY_SPIN, spin_iters=_iters(case, seed), out=s["out"],
                                       tile=(case["tile_w"], case["tile_h"]), inputs=inputs)
    return s


def _csr_buffers(n, edges):
    """Room for a graph's CSR, the columns at most `edges` (random rectangles have 20 to 25 a launch)."""
    size = dict(row_ptr=n + 1, col=edges, indeg=n)
    return {k: torch.full((m,), -1, dtype=torch.int32, device="cuda") for k, m in size.items()}


def _csr(handle, into):
    """The analysed graph's CSR in the program's device buffers."""
    if grt.rt_graph_stats(handle)["n_edges"] > into["col"].numel():
        raise ValueError("more edges than the column buffer holds")
    status = grt.load().rt_copy_csr(handle, *[into[k].data_ptr() for k in ("row_ptr", "col", "indeg")])
    if status != grt.RT_OK:
        raise grt.GrtError(status, grt.rt_last_error())
    return into


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "call":
        g = state["graph"]
        state["state"].copy_(state["start"])
        g.clear()
        g.launch(*state["launches"])
        g.analyze()
        g.execute()
        g.sync()
        return state["state"]
    if kind == "analyze":
        g = state["graph"]
        g.clear()
        g.launch(*state["launches"])
        g.analyze()
        return _csr(g.h, state["csr"])
    if kind == "execute":
        state["graph"].execute()
        return state["out"]
    if kind == "replay":
        if "state" in state:
            state["state"].copy_(state["start"])
        state["graph"].replay(case["replays"])
        return state["state"] if "state" in state else state["out"]
    if kind == "stitch":
        state["graph"].execute_stitched(case["replays"])
        return state["out"]
    if kind == "capture":
        b = grt.Batch.capture(state["traces"], body=grt.RT_BODY_SPIN, spin_iters=state["iters"], out=state["out"],
                              tile=(case["tile_w"], case["tile_h"]), inputs=state["inputs"])
        b.execute(1)
        b.sync()
        csr = _csr(b.graph_h, state["csr"])
        b.close()
        return dict(csr, out=state["out"])
    state["batch"].execute(case["replays"], blocks=case["blocks"], warps=case["warps"], claim=case["claim"],
                           keep=case["keep"])
    return state["out"]


# ----------------------------------------------------------------------------------------------------------------
def _grid_edges(pattern, width, steps):
    k = {"stencil": 3 * width - 2, "butterfly": 2 * width, "random": min(5, width) * width}[pattern]
    return (steps - 1) * k


def work(case):
    kind = case["kind"]
    iters = case.get("iters", 0) + 4  # the seed adds 0..7
    if kind == "call" or case.get("trace") == "stencil_1d":
        n = case["pieces"] * case["steps"]
        e = 2 * (case["pieces"] - 1) * case["steps"]  # its read and its write neighbours, a little over
        if kind == "call":  # launches in, state out; the DAG in between need not leave the chip
            return {"bytes": 4 * n + 2 * 17 * n + 4 * n + 8 * case["pieces"], "flops": n}
        return {"bytes": 12 * n + 4 * e + 8 * case["pieces"], "flops": n * case["replays"]}
    if kind == "analyze":
        if case["trace"] == "rects":
            n, r, per = case["n"], 2.5 * case["n"], case["bounds"] // 2 + 1
            return {"bytes": 4 * n + per * r + 8 * n + 4 * 20 * n, "flops": 0}  # about 20 edges a launch
        w, t = case["width"], case["steps"]
        n, e = w * t, _grid_edges("random", w, t)
        into = (case["bounds"] // 2 + 1) * (e + n) if case["encode"] == "region" else 4 * n + 4 * e
        return {"bytes": 4 * n + into + 8 * n + 4 * e, "flops": 0}
    if kind in ("execute", "replay", "stitch"):
        w, t, rep = case["width"], case["steps"], case.get("replays", 1)
        n, e = w * t, _grid_edges(case["pattern"], w, t)
        outs = rep if kind == "stitch" else 1
        return {"bytes": 8 * n + 4 * e + 4 * n * outs, "flops": 2 * iters * n * rep}
    mean = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])  # of the log-uniform task count
    n = mean * case["graphs"]
    if kind == "capture":
        return {"bytes": 4 * n + 33 * 2.5 * n + 8 * n + 4 * 20 * n + 4 * n, "flops": 24 * n}
    return {"bytes": 8 * n + 4 * 3.3 * n + 4 * n, "flops": 2 * iters * n * case["replays"]}


def _spin(ids, iters):
    x = ids.astype(np.uint64)
    for _ in range(iters):
        x = (x * np.uint64(1664525) + np.uint64(1013904223)) & np.uint64(0xFFFFFFFF)
    return x.astype(np.uint32).view(np.int32)


def exact(case, seed):
    kind = case["kind"]
    if kind == "call" or case.get("body") == "COUNTER":  # every task adds one to its piece's counter
        g = np.random.Generator(np.random.PCG64(seed))
        start = g.integers(-1 << 31, 1 << 31, size=case["pieces"], dtype=np.int64)
        return (start + case["steps"] * case.get("replays", 1)).astype(np.uint32).view(np.int32)
    if kind in ("execute", "replay") and case["body"] == "SPIN":
        return _spin(np.arange(case["width"] * case["steps"]), _iters(case, seed))
    if kind == "stitch":
        return np.tile(_spin(np.arange(case["width"] * case["steps"]), _iters(case, seed)), case["replays"])
    if kind == "batch":  # a batched body sees its own graph's task ids
        return _spin(np.concatenate([np.arange(w * t) for w, t, _, _ in _batch_specs(case, seed)]), _iters(case, seed))
    if kind == "analyze" and case["trace"] == "taskbench":  # task (i, t) follows its predecessor columns of step t - 1
        w, t = case["width"], case["steps"]
        n, pc = w * t, tg.taskbench_preds(w, t, "random", seed)
        src = (pc + (np.arange(t - 1) * w)[:, None, None]).reshape(-1)
        dst = np.repeat(np.arange(w, n), pc.shape[2])
        order = np.argsort(src * n + dst, kind="stable")
        row_ptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
        return dict(row_ptr=row_ptr.astype(np.int32), col=dst[order].astype(np.int32),
                    indeg=np.bincount(dst, minlength=n).astype(np.int32))
    return None  # random rectangles have no closed form; a fused multiply-add has none in numpy
