"""Performance cases: the calls a program makes through this library's public
entry points (include/igs.h and its binding), from single box copies to whole
programs that are lowered, executed and read back.

A case's "kind" says which entry point it goes through:
  copy    igs_box_copy on device memory the caller owns
  static  igs_lower_static: a whole program into the caller's device arrays
  run     one program's life: context, buffers with host data, submissions,
          lowering and execution (igs_run, or plain submissions and
          igs_execute), the instruction graphs and the buffers' contents
  batch   many independent programs lowered in one launch (igs_lower_batch)
  serve   many program streams lowered by the device-resident request loop
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2503_10516_gb300 import igs
from paper_2503_10516_gb300 import workloads as W

WINDOW = 16       # igs_run: submissions per executor window, as the benchmark uses
BATCH_POOL = 96   # programs a batch is chosen from


def listed():
    return [
        # halo rows of a time step of the 8192-wide wave program: many short
        # contiguous copies, the smallest call there is
        {"name": "copy_halo", "kind": "copy", "jobs": 24, "planes": 1, "rows": 1, "cols": 8192, "src_pad": 0,
         "dst_pad": 0, "off": 0, "elem": 4},
        # a growing allocation moves: 512 MiB into a wider row pitch (the benchmark's resize copy)
        {"name": "copy_resize", "kind": "copy", "jobs": 1, "planes": 1, "rows": 8192, "cols": 16384, "src_pad": 0,
         "dst_pad": 64, "off": 0, "elem": 4},
        # sub-boxes of 3D allocations with odd extents: no row starts on a 16-byte boundary
        {"name": "copy_ragged", "kind": "copy", "jobs": 3, "planes": 13, "rows": 411, "cols": 1003, "src_pad": 6,
         "dst_pad": 19, "off": 3, "elem": 4},
        # a runtime that cannot allocate lowers two dozen wave steps with a probe now and then
        {"name": "static_wave", "kind": "static", "program": "wave", "n": 8192, "steps": 24, "nodes": 4, "devices": 4,
         "chunks": 64, "lookahead": 8, "horizon": 4},
        # the small Jacobi configuration, one lowering launch per task: latency
        {"name": "run_jacobi_small", "kind": "run", "program": "jacobi", "n": 256, "steps": 8, "nodes": 2,
         "devices": 2, "chunks": 4, "lookahead": 0, "horizon": 4, "mode": "plain", "executor": 0},
        # the headline: wave stencil on 4 x 4 devices, lowering and execution overlapped
        {"name": "run_wave", "kind": "run", "program": "wave", "n": 4096, "steps": 192, "nodes": 4, "devices": 4,
         "chunks": 64, "lookahead": 8, "horizon": 4, "mode": "run", "executor": 0},
        # few devices and a large grid: the stencil itself is the work
        {"name": "run_jacobi_large", "kind": "run", "program": "jacobi", "n": 8192, "steps": 400, "nodes": 1,
         "devices": 4, "chunks": 8, "lookahead": 8, "horizon": 4, "mode": "run", "executor": 0},
        # all-pairs N-body on 8 x 4 devices: every position to every node, then 2^32 body pairs a step
        {"name": "run_nbody", "kind": "run", "program": "nbody", "n": 1 << 16, "steps": 6, "nodes": 8, "devices": 4,
         "chunks": 128, "lookahead": 4, "horizon": 4, "mode": "run", "executor": 0},
        # growing rows without lookahead: every task reallocates and copies what there is
        {"name": "run_grow", "kind": "run", "program": "grow", "n": 4096, "cols": 4096, "steps": 1, "nodes": 1,
         "devices": 2, "chunks": 2, "lookahead": 0, "horizon": 4, "mode": "run", "executor": 0},
        # 3D integer fields with odd extents on the out-of-order executor
        {"name": "run_field_flow", "kind": "run", "program": "field", "n": 193, "steps": 24, "nodes": 2, "devices": 3,
         "chunks": 13, "lookahead": 4, "horizon": 4, "mode": "run", "executor": 1},
        # a batch of uneven programs in one launch
        {"name": "batch", "kind": "batch", "programs": 24, "percent": 5},
        # streams of growing-row tasks through the served loop
        {"name": "serve", "kind": "serve", "streams": 16, "rows": 2048, "lookahead": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["copy", "copy", "static", "run", "run", "run", "run", "batch", "serve"])
    if kind == "copy":
        elem = rng.choice([1, 2, 4, 4, 8, 16])
        total = _log(rng, 1 << 15, 1 << 29) // elem
        jobs = rng.choice([1, 1, 2, 5, 16, 32])
        planes = rng.choice([1, 1, 3, 17])
        cols = max(1, min(_log(rng, 64, 16384), total // (jobs * planes)))
        rows = max(1, total // (jobs * planes * cols))
        pad = rng.choice([0, 0, 1, 16, 64])
        return {"kind": "copy", "jobs": jobs, "planes": planes, "rows": rows, "cols": cols,
                "src_pad": rng.choice([0, pad, 7]), "dst_pad": pad, "off": rng.randint(0, pad), "elem": elem}
    if kind == "static":
        nodes = rng.choice([1, 2, 4, 8])
        devices = rng.choice([1, 2, 4])
        return {"kind": "static", "program": rng.choice(["wave", "jacobi", "nbody"]), "n": _log(rng, 200, 8192),
                "steps": rng.randint(4, 24), "nodes": nodes, "devices": devices,
                "chunks": nodes * devices * rng.choice([1, 2, 4]), "lookahead": rng.choice([0, 2, 8]),
                "horizon": rng.choice([2, 4])}
    if kind == "batch":
        return {"kind": "batch", "programs": rng.randint(4, 24), "percent": rng.choice([2, 3, 5])}
    if kind == "serve":
        return {"kind": "serve", "streams": rng.randint(2, 16), "rows": _log(rng, 200, 2048),
                "lookahead": rng.choice([0, 8, 0xFFFFFFFF])}
    program = rng.choice(["wave", "wave", "jacobi", "jacobi", "nbody", "grow", "field"])
    nodes, devices = rng.choice([(1, 2), (1, 4), (2, 2), (2, 3), (4, 4)])
    case = {"kind": "run", "program": program, "steps": 1, "nodes": nodes, "devices": devices,
            "chunks": nodes * devices * rng.choice([1, 2, 3]) + rng.randint(0, 1), "lookahead": rng.choice([0, 4, 8]),
            "horizon": 4, "mode": rng.choice(["run", "run", "run", "plain"]), "executor": rng.choice([0, 0, 1])}
    if program in ("wave", "jacobi"):
        case.update(n=_log(rng, 150, 6000), steps=_log(rng, 4, 120))
    elif program == "nbody":
        case.update(n=_log(rng, 1000, 60000), steps=rng.randint(1, 4))
    elif program == "grow":
        case.update(n=_log(rng, 200, 3000), cols=_log(rng, 16, 4096), nodes=1, devices=2, chunks=2)
    else:
        case.update(n=rng.randint(20, 180), steps=rng.randint(3, 24))
    return case


# ---- programs ----------------------------------------------------------------


class PackedTask:
    """A task whose descriptor words a program has laid out once."""

    def __init__(self, task):
        self.words = np.ascontiguousarray(task.flat(), dtype=np.uint32)
        self.chunks, self.accessors = task.chunks, task.accessors

    def flat(self):
        return self.words


def _field_program(case, rng):
    """Two 3D integer fields and a 3D coefficient field: each step writes one
    field from the other's neighbourhood and the coefficients of the item's plane."""
    n = case["n"]
    ext = (n, n - 2, n + 3)
    init = lambda: rng.integers(0, 2**32, size=ext, dtype=np.uint32)  # noqa: E731
    ops = [("buffer", W.Buffer(3, ext, 4, init(), "u32")), ("buffer", W.Buffer(3, ext, 4, None, "u32")),
           ("buffer", W.Buffer(3, ext, 4, init(), "u32"))]
    src, dst = 0, 1
    for k in range(case["steps"]):
        coef = W.one_to_one() if k % 3 else W.row_slice()
        ops.append(("task", W.Task(3, ext, case["chunks"], W.K_GENERIC,
                                   [W.Accessor(dst, W.WRITE, W.one_to_one()),
                                    W.Accessor(src, W.READ, W.neighborhood(1)), W.Accessor(2, W.READ, coef)])))
        src, dst = dst, src
    return W.Program("field", case["nodes"], case["devices"], case["horizon"], case["lookahead"], ops + [("flush",)])


def _program(case, seed):
    c, rng = case, np.random.default_rng(seed)
    shape = dict(nodes=c["nodes"], devices=c["devices"], chunks=c["chunks"], lookahead=c["lookahead"],
                 horizon_step=c["horizon"])
    if c["program"] == "wave":
        return W.wave_program(n=c["n"], steps=c["steps"], seed=seed, **shape)
    if c["program"] == "jacobi":
        return W.jacobi_program(n=c["n"], steps=c["steps"], seed=seed, **shape)
    if c["program"] == "nbody":
        return W.nbody_program(n=c["n"], steps=c["steps"], seed=seed, **shape)
    if c["program"] == "grow":
        return W.growing_program(rows_max=c["n"], cols=c["cols"], seed=seed, **shape)
    return _field_program(c, rng)


def _shape_program(case, seed):
    """A program for lowering alone (which never reads buffer values): the
    steps of the case, and every sixth step a probe that reads a window of the
    newest field at a place drawn from the seed."""
    c, rng = case, np.random.default_rng(seed)
    small = dict(case, n=8 if c["program"] != "nbody" else c["chunks"])
    prog = _program(small, 1)
    ops, step = [], 0
    for op in prog.ops:
        if op[0] == "buffer":
            ext = (c["n"], c["n"], 1) if op[1].dims == 2 else (c["n"], 1, 1)
            ops.append(("buffer", W.Buffer(op[1].dims, ext, op[1].elem_size, op[1].init, op[1].dtype)))
        elif op[0] == "task":
            t = op[1]
            t.range = (c["n"], c["n"], 1) if t.dims == 2 else (c["n"], 1, 1)
            ops.append(op)
            step += 1
            if step % 6 == 0:
                lo = [int(rng.integers(0, c["n"] - 16)) for _ in range(t.dims)]
                read = W.fixed_box(lo, [v + 16 for v in lo])
                ops.append(("task", W.Task(t.dims, (16, 16 if t.dims == 2 else 1, 1), 1, W.K_NOP,
                                           [W.Accessor(t.accessors[-1].buffer, W.READ, read),
                                            W.Accessor(len(prog.buffers), W.WRITE, W.one_to_one())])))
        else:
            ops.append(op)
    t = prog.tasks[0]
    probe = W.Buffer(t.dims, (16, 16, 1) if t.dims == 2 else (16, 1, 1), prog.buffers[0].elem_size, None)
    at = sum(op[0] == "buffer" for op in ops)
    return W.Program(prog.name, prog.nodes, prog.devices, prog.horizon_step, prog.lookahead,
                     ops[:at] + [("buffer", probe)] + ops[at:])


def _packed(prog):
    ops = [("task", PackedTask(op[1])) if op[0] == "task" else op for op in prog.ops]
    return W.Program(prog.name, prog.nodes, prog.devices, prog.horizon_step, prog.lookahead, ops)


def _caps(prog):
    """Context capacities a program of this shape needs, with room to spare."""
    tasks = prog.tasks
    chunks = max(t.chunks for t in tasks)
    per_node = -(-chunks // prog.nodes)
    instrs = len(tasks) * (6 * per_node + 8 * prog.nodes + 48) + 1024
    return {"max_instructions": instrs, "max_edges": 24 * instrs, "max_boxes": 8 * instrs, "map_heap": 1 << 17,
            "scratch_capacity": 8192, "max_buffers": max(1, len(prog.buffers)), "max_live_allocs": 1024,
            "max_allocations": 1 << 15, "max_queue": max(256, 2 * len(prog.ops) + 16)}


def _context(prog, mode, caps):
    ctx = igs.Context(prog.nodes, prog.devices, prog.horizon_step, prog.lookahead, mode=mode, **caps)
    for b in prog.buffers:
        ctx.create_buffer(b.dims, b.extent[:b.dims], b.elem_size, b.init)
    return ctx


def _submit(ctx, prog):
    for op in prog.ops:
        if op[0] == "task":
            ctx.submit(op[1])
        elif op[0] == "flush":
            ctx.submit_epoch()


RECORDS = (("instrs", 11), ("edges", 3), ("boxes", 6), ("binds", 7), ("diags", 3))  # 32-bit words of a record


def _graph_arrays(case):
    """Host arrays that the graphs of all nodes are fetched into, one after the
    other: as large as any program of the case needs."""
    c = case
    if c["kind"] == "batch":
        total, nodes = 6000 * c["programs"] * c["percent"], 32 * c["programs"]
    elif c["kind"] == "serve":
        total, nodes = c["streams"] * (2 * c["rows"] + 64), c["streams"]
    else:
        tasks = {"nbody": 2 * c["steps"], "grow": c["n"] // 16}.get(c["program"], c["steps"])
        nodes = c["nodes"]
        total = nodes * (tasks * (4 * -(-c["chunks"] // nodes) + 4 * nodes + 24) + 256)
    rows = {"instrs": total, "edges": 8 * total, "boxes": 3 * total, "binds": 2 * total, "diags": 4096}
    return {**{k: np.zeros((rows[k], w), np.int32) for k, w in RECORDS}, "counts": np.zeros((nodes, 5), np.int32)}


def _fetch(ctxs, progs, arrays):
    """Every node's graph into the arrays; counts has each node's records."""
    at, view, row = [0] * len(RECORDS), igs.GraphView(), 0
    ptr_cap_num = (("instrs", "instr_cap", "num_instrs"), ("edges", "edge_cap", "num_edges"),
                   ("boxes", "box_cap", "num_boxes"), ("binds", "bind_cap", "num_binds"),
                   ("diags", "diag_cap", "num_diags"))
    for ctx, prog in zip(ctxs, progs):
        for n in range(prog.nodes):
            view.node = n
            for k, (name, cap, _) in enumerate(ptr_cap_num):
                a = arrays[name]
                setattr(view, name, a.ctypes.data + at[k] * a.strides[0])
                setattr(view, cap, len(a) - at[k])
            r = igs.lib().igs_fetch_instructions(ctx.handle, ctypes.byref(view))
            if r != igs.IGS_OK:
                raise igs.IgsError(r, "fetch_instructions")
            for k, (_, _, num) in enumerate(ptr_cap_num):
                got = getattr(view, num)
                arrays["counts"][row, k] = got
                at[k] += got
            row += 1
    return arrays


# ---- prepare / run -------------------------------------------------------------


def _prepare_copy(case, seed):
    c, dev = case, torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    src_cols, dst_cols = c["cols"] + c["src_pad"], c["cols"] + c["dst_pad"]
    src_at, dst_at = min(c["off"], c["src_pad"]), min(c["off"], c["dst_pad"])
    jobs = (igs.CopyJob * c["jobs"])()
    srcs, dsts = [], []
    for j in range(c["jobs"]):
        src = torch.randint(0, 256, (c["planes"] * c["rows"] * src_cols * c["elem"],), dtype=torch.uint8, device=dev,
                            generator=gen)
        dst = torch.zeros(c["planes"] * c["rows"] * dst_cols * c["elem"], dtype=torch.uint8, device=dev)
        srcs.append(src)
        dsts.append(dst)
        # one coordinate system for both: the copied box starts at column 64
        jobs[j].src, jobs[j].dst, jobs[j].elem_size = src.data_ptr(), dst.data_ptr(), c["elem"]
        for box, lo, cols in ((jobs[j].src_box, 64 - src_at, src_cols), (jobs[j].dst_box, 64 - dst_at, dst_cols),
                              (jobs[j].box, 64, c["cols"])):
            box.lo[:] = (0, 0, lo)
            box.hi[:] = (c["planes"], c["rows"], lo + cols)
    return {"kind": "copy", "jobs": jobs, "n": c["jobs"], "src": srcs, "dst": dsts}


def _prepare_static(case, seed):
    prog = _shape_program(case, seed)
    caps = _caps(prog)
    ni = caps["max_instructions"]
    sizes = {"instrs": (ni, 11), "edges": (12 * ni, 3), "boxes": (4 * ni, 6), "binds": (2 * ni, 7), "diags": (256, 3)}
    outs, arr = [], (igs.StaticOutput * prog.nodes)()
    for n in range(prog.nodes):
        o = {k: torch.zeros(s, dtype=torch.int32, device="cuda") for k, s in sizes.items()}
        o["counts"] = torch.zeros(6, dtype=torch.int32, device="cuda")
        for k, cap in (("instrs", "instr_cap"), ("edges", "edge_cap"), ("boxes", "box_cap"), ("binds", "bind_cap"),
                       ("diags", "diag_cap")):
            setattr(arr[n], k, o[k].data_ptr())
            setattr(arr[n], cap, sizes[k][0])
        arr[n].counts = o["counts"].data_ptr()
        outs.append(o)
    bufs, tasks = prog.buffers, prog.tasks
    sb = (igs.StaticBuffer * len(bufs))()
    for i, b in enumerate(bufs):
        sb[i].dims, sb[i].elem_size, sb[i].has_init = b.dims, b.elem_size, int(b.init is not None)
        sb[i].extent[:] = b.extent
    words = np.concatenate([t.flat() for t in tasks])
    ops, nb, nt = [], 0, 0
    for op in prog.ops:
        if op[0] == "buffer":
            ops.append((0, nb))
            nb += 1
        elif op[0] == "task":
            ops.append((1, nt))
            nt += 1
        else:
            ops.append((2, 0))
    so = (igs.StaticOp * len(ops))(*[igs.StaticOp(k, a) for k, a in ops])
    cfg = igs.Config(num_nodes=prog.nodes, devices_per_node=prog.devices, horizon_step=prog.horizon_step,
                     lookahead=prog.lookahead)
    return {"kind": "static", "cfg": cfg, "bufs": sb, "nb": nb, "words": words, "nt": nt, "ops": so, "no": len(ops),
            "arr": arr, "outs": outs}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "copy":
        return _prepare_copy(case, seed)
    if kind == "static":
        return _prepare_static(case, seed)
    if kind == "run":
        prog = _packed(_program(case, seed))
        caps = _caps(prog)
        return {"kind": "run", "prog": prog, "caps": caps, "plain": case["mode"] == "plain",
                "executor": case["executor"], "dtype": np.int32 if case["program"] == "field" else np.float32,
                "graph": _graph_arrays(case)}
    rng = np.random.default_rng(seed)
    if kind == "batch":
        # programs of the uneven batch at a share of their tasks; the seed says which of them
        pool = W.batch_programs(count=BATCH_POOL, scale=case["percent"] / 100.0)
        chosen = rng.permutation(BATCH_POOL)[:case["programs"]]
        progs = [_packed(pool[i]) for i in sorted(int(v) for v in chosen)]
    else:
        progs = [_packed(W.growing_program(rows_max=case["rows"], cols=int(rng.choice([1, 2048, 8192])), devices=2,
                                           chunks=2, lookahead=case["lookahead"], seed=seed * 1000 + i))
                 for i in range(case["streams"])]
    return {"kind": kind, "progs": progs, "caps": [_caps(p) for p in progs], "graph": _graph_arrays(case)}


def _run_program(state):
    prog = state["prog"]
    ctx = _context(prog, igs.MODE_PLAIN if state["plain"] else igs.MODE_BATCHED, state["caps"])
    ctx.set_executor(state["executor"])
    _submit(ctx, prog)
    if state["plain"]:
        ctx.sync()
        ctx.execute()
    else:
        ctx.run(WINDOW)
    out = {"graph": _fetch([ctx], [prog], state["graph"]),
           "buffers": [ctx.read_buffer(i, (0, 0, 0), b.extent, b.elem_size).view(state["dtype"])
                       for i, b in enumerate(prog.buffers)]}
    ctx.close()
    return out


def _run_batch(state):
    ctxs = [_context(p, igs.MODE_BATCHED, caps) for p, caps in zip(state["progs"], state["caps"])]
    for ctx, p in zip(ctxs, state["progs"]):
        _submit(ctx, p)
    igs.lower_batch(ctxs)
    out = _fetch(ctxs, state["progs"], state["graph"])
    for ctx in ctxs:
        ctx.close()
    return out


def _run_serve(state):
    progs = state["progs"]
    server = igs.Server(max_slots=len(progs))
    ctxs = [_context(p, igs.MODE_BATCHED, caps) for p, caps in zip(progs, state["caps"])]
    for ctx, p in zip(ctxs, progs):
        if server.attach(ctx, 2 * len(p.ops) + 16) != igs.IGS_OK:
            raise RuntimeError("a stream was not admitted")
    server.start()
    # submissions arrive interleaved, one of every stream at a time
    feeds = [[op for op in p.ops if op[0] != "buffer"] for p in progs]
    for k in range(max(len(f) for f in feeds)):
        for ctx, feed in zip(ctxs, feeds):
            if k < len(feed):
                if feed[k][0] == "task":
                    ctx.submit(feed[k][1])
                else:
                    ctx.submit_epoch()
    for ctx in ctxs:
        server.detach(ctx)
    server.stop()
    out = _fetch(ctxs, progs, state["graph"])
    for ctx in ctxs:
        ctx.close()
    server.close()
    return out


def run(state):
    kind = state["kind"]
    if kind == "copy":
        r = igs.lib().igs_box_copy(state["jobs"], state["n"], torch.cuda.current_stream().cuda_stream)
        if r != igs.IGS_OK:
            raise igs.IgsError(r, "box_copy")
        return state["dst"]
    if kind == "static":
        s = state
        r = igs.lib().igs_lower_static(ctypes.byref(s["cfg"]), s["bufs"], s["nb"],
                                       s["words"].ctypes.data_as(ctypes.POINTER(ctypes.c_uint32)), s["nt"], s["ops"],
                                       s["no"], s["arr"], torch.cuda.current_stream().cuda_stream)
        if r != igs.IGS_OK:
            raise igs.IgsError(r, "lower_static")
        return s["outs"]
    if kind == "run":
        return _run_program(state)
    return _run_batch(state) if kind == "batch" else _run_serve(state)


# ---- work and exact values --------------------------------------------------------


def _graph_bytes(tasks, chunks, nodes):
    """Records of a lowered task: per chunk a kernel instruction (44 bytes)
    with its edges (three of 12), box (24) and bindings (two of 28); per node
    a handful of transfers."""
    return tasks * (chunks * (44 + 36 + 24 + 56) + nodes * 4 * (44 + 24 + 24) + igs.TASK_WORDS * 4)


def work(case):
    c, kind = case, case["kind"]
    if kind == "copy":
        return {"bytes": 2.0 * c["jobs"] * c["planes"] * c["rows"] * c["cols"] * c["elem"], "flops": 0.0}
    if kind == "batch":
        return {"bytes": float(c["programs"] * _graph_bytes(10 * c["percent"], 64, 6)), "flops": 0.0}
    if kind == "serve":
        return {"bytes": float(c["streams"] * _graph_bytes(c["rows"] / 32.5, 2, 1)), "flops": 0.0}
    n, steps = c["n"], c["steps"]
    tasks = {"nbody": 2 * steps, "grow": n / 32.5}.get(c["program"], steps)
    graph = float(_graph_bytes(tasks, c["chunks"], c["nodes"]))
    if kind == "static":
        return {"bytes": graph, "flops": 0.0}
    # every kernel's inputs read once and outputs written once
    data, flops = {"wave": (12.0 * n * n * steps, 9.0 * n * n * steps),
                   "jacobi": (8.0 * n * n * steps, 4.0 * n * n * steps),
                   "nbody": (96.0 * n * steps, 20.0 * n * n * steps),
                   "grow": (4.0 * n * c.get("cols", 1) * 2, 2.0 * n * c.get("cols", 1)),
                   "field": (12.0 * n * (n - 2) * (n + 3) * steps, 0.0)}[c["program"]]
    return {"bytes": graph + data, "flops": flops}


def _stencil_step(u, prev):
    """One step on the interior (borders keep u): the wave update, or Jacobi's without prev."""
    out = u.clone()
    n, s, w, e = u[:-2, 1:-1], u[2:, 1:-1], u[1:-1, :-2], u[1:-1, 2:]
    if prev is None:
        out[1:-1, 1:-1] = (n + s + w + e) * 0.25
    else:
        c = u[1:-1, 1:-1]
        out[1:-1, 1:-1] = 2.0 * c - prev[1:-1, 1:-1] + 0.25 * (n + s + w + e - 4.0 * c)
    return out


def _nbody(p, v, steps):
    dt = float(np.float32(0.01))
    eps = float(np.float32(1e-6))
    for _ in range(steps):
        x, w, acc = p[:, :3], p[:, 3], torch.empty_like(p[:, :3])
        for i in range(0, len(p), 1024):
            d = x[None, :, :] - x[i:i + 1024, None, :]
            r2 = (d * d).sum(2) + eps
            acc[i:i + 1024] = (d * (w[None, :] / (r2 * r2.sqrt()))[:, :, None]).sum(1)
        v[:, :3] += acc * dt
        p[:, :3] += v[:, :3] * dt
    return p, v


def exact(case, seed):
    c = case
    if c["kind"] != "run" or c["program"] == "field":
        return None  # whole numbers
    prog = _program(c, seed)
    init = [None if b.init is None else torch.from_numpy(b.init).cuda().double() for b in prog.buffers]
    if c["program"] == "nbody":
        bufs = [t[:, None, None, :] for t in _nbody(init[0], init[1], c["steps"])]
    elif c["program"] == "grow":
        rows, cols = c["n"], c["cols"]
        buf = torch.empty(rows, cols, dtype=torch.float64, device="cuda")
        first = prog.tasks[0].range[0]
        y, x = torch.arange(rows, device="cuda")[:, None], torch.arange(cols, device="cuda")[None, :]
        buf[:first] = ((y[:first] * 131 + x * 7) & 1023).double() * 0.5
        for t in prog.tasks[1:]:
            r = t.params[0]
            buf[r:r + t.range[0]] = buf[r - 1] * 0.5 + (y[r:r + t.range[0]] & 255).double()
        bufs = [buf[:, :, None, None]]
    else:
        ring = init
        for k in range(c["steps"]):
            if c["program"] == "wave":
                prev, cur, nxt = k % 3, (k + 1) % 3, (k + 2) % 3
                ring[nxt] = _stencil_step(ring[cur], ring[prev])
            else:
                ring[(k + 1) % 2] = _stencil_step(ring[k % 2], None)
        if any(t is None for t in ring):
            return None
        bufs = [t[:, :, None, None] for t in ring]
    return {"graph": None, "buffers": bufs}
