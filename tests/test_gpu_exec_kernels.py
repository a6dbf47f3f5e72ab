"""GPU: the execution kernels at the sizes where their tiles, lanes and
vector widths change, against the same operations in numpy (bit for bit: both
round after every operation, in the same order)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2503_10516_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(prog, executor):
    from paper_2503_10516_gb300 import igs
    c = igs.Context(prog.nodes, prog.devices, prog.horizon_step, prog.lookahead, mode=igs.MODE_BATCHED)
    c.set_executor(executor)
    for b in prog.buffers:
        c.create_buffer(b.dims, b.extent[:b.dims], b.elem_size, b.init)
    for t in prog.tasks:
        c.submit(t)
    c.flush()
    c.execute()
    return c


def _nbody_velocity(P, V, i):
    """Body i's velocity after one step: the terms in index order, float32."""
    eps, dt = np.float32(1e-6), np.float32(0.01)
    with np.errstate(all="ignore"):
        dx, dy, dz = P[:, 0] - P[i, 0], P[:, 1] - P[i, 1], P[:, 2] - P[i, 2]
        r2 = ((dx * dx + dy * dy) + dz * dz) + eps
        wgt = P[:, 3] * (np.float32(1.0) / (r2 * np.sqrt(r2)))
        v = V[i].copy()
        for c, d in enumerate((dx, dy, dz)):
            v[c] = v[c] + np.add.accumulate(d * wgt, dtype=np.float32)[-1] * dt
    return v


@pytest.mark.parametrize("executor", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 255, 257, 1000, 9727, 9729, 117001])
@pytest.mark.parametrize("far", [False, True])
def test_nbody_step_tiles(n, far, executor):
    """One N-body step around the tile sizes and the changes of the lanes per
    body (9728 and 116736 bodies on 152 SMs). far: bodies at equal places, so
    far away that the squared distance leaves the fast range or overflows,
    and at infinity."""
    prog = W.nbody_program(n=n, steps=1, nodes=1, devices=2, chunks=3, lookahead=0, seed=n)
    prog.ops = [op for op in prog.ops if op[0] != "task"][:2] + [("task", prog.tasks[0]), ("flush",)]
    P, V = prog.buffers[0].init, prog.buffers[1].init
    P[:, 3] = np.linspace(-1, 2, n, dtype=np.float32)
    if far:
        P[n // 2] = P[0]
        for k, x in enumerate((3e11, -1e13, 2e19, np.inf)):
            P[(7 + 61 * k) % n, k % 3] = np.float32(x)
    c = _run(prog, executor)
    got = c.read_buffer(1, (0, 0, 0), (n, 1, 1), 16).view(np.float32).reshape(n, 4)
    c.close()
    for i in sorted({0, n // 3, n // 2, n - 1, min(n - 1, 63), min(n - 1, 64)} | {(7 + 61 * k) % n for k in range(4)}):
        assert np.array_equal(got[i], _nbody_velocity(P, V, i), equal_nan=True), (n, i)


def _stencil_reference(prog):
    """The stencil program's buffers, step by step in float32."""
    bufs = [None if b.init is None else b.init.astype(np.float32).copy() for b in prog.buffers]
    for t in prog.tasks:
        ids = [a.buffer for a in t.accessors]
        u = bufs[ids[-2]]
        out = u.copy()
        if min(u.shape) > 2:
            n, s, w, e, c = u[:-2, 1:-1], u[2:, 1:-1], u[1:-1, :-2], u[1:-1, 2:], u[1:-1, 1:-1]
            t5 = (n + s) + (w + e)
            if len(ids) == 2:
                out[1:-1, 1:-1] = t5 * np.float32(0.25)
            else:
                t2 = np.float32(2.0) * c - bufs[ids[0]][1:-1, 1:-1]
                out[1:-1, 1:-1] = t2 + np.float32(0.25) * (t5 - np.float32(4.0) * c)
        bufs[ids[-1]] = out
    return bufs


@pytest.mark.parametrize("executor", [0, 1])
@pytest.mark.parametrize("kind", ["jacobi", "wave"])
@pytest.mark.parametrize("shape", [(1, 1), (3, 2), (5, 127), (4, 128), (40, 129), (33, 131), (65, 256), (70, 260),
                                   (130, 516), (37, 1028), (19, 1031), (513, 2052)], ids=str)
@pytest.mark.parametrize("chunks", [1, 5, (2 << 16) | 3])
def test_stencil_strips(shape, chunks, kind, executor):
    """Stencil strips at ragged and vector widths, heights around the tiles'
    rows, splits along rows and along both dimensions (whose allocations start
    at any column), three steps."""
    make = W.jacobi_program if kind == "jacobi" else W.wave_program
    prog = make(n=4, steps=3, nodes=1, devices=2, chunks=chunks, lookahead=0)
    rng = np.random.default_rng(shape[0] * 4096 + shape[1])
    for b in prog.buffers:
        b.extent = (*shape, 1)
        if b.init is not None:
            b.init = rng.random(shape, dtype=np.float32)
    for t in prog.tasks:
        t.range = (*shape, 1)
    want = _stencil_reference(prog)
    c = _run(prog, executor)
    for i, w in enumerate(want):
        got = c.read_buffer(i, (0, 0, 0), (*shape, 1), 4).view(np.float32).reshape(shape)
        assert np.array_equal(got, w), (shape, i)
    c.close()
