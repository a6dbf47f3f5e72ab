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


def _copy_case(torch, rng, n_jobs, elem, ext, pads, offs):
    """n_jobs copies of a box of extent ext between allocations that are wider
    by pads (source, destination) per dimension, their first bytes off by offs."""
    from paper_2503_10516_gb300 import igs
    jobs, want, keep = (igs.CopyJob * n_jobs)(), [], []
    for j in range(n_jobs):
        arrs = []
        for k in range(2):
            shape = [e + p for e, p in zip(ext, pads[k])]
            host = rng.integers(0, 256, size=int(np.prod(shape)) * elem, dtype=np.uint8)
            dev = torch.zeros(len(host) + 16, dtype=torch.uint8, device="cuda")
            dev[offs[k]:offs[k] + len(host)] = torch.from_numpy(host).cuda()
            arrs.append((host.reshape(*shape, elem), dev, shape))
        (src, sdev, ss), (dst, ddev, ds) = arrs
        jobs[j].src, jobs[j].dst, jobs[j].elem_size = sdev.data_ptr() + offs[0], ddev.data_ptr() + offs[1], elem
        for box, shape, pad in ((jobs[j].src_box, ss, pads[0]), (jobs[j].dst_box, ds, pads[1]), (jobs[j].box, ext, (0,) * 3)):
            lo = [100 - p // 2 for p in pad]
            box.lo[:], box.hi[:] = lo, [v + s for v, s in zip(lo, shape)]
        at = [tuple(slice(p // 2, p // 2 + e) for p, e in zip(pad, ext)) for pad in pads]
        dst[at[1]] = src[at[0]]
        keep.append((sdev, ddev))
        want.append(dst.reshape(-1))
    r = igs.lib().igs_box_copy(jobs, n_jobs, torch.cuda.current_stream().cuda_stream)
    assert r == igs.IGS_OK
    for (_, ddev), w in zip(keep, want):
        got = ddev.cpu().numpy()
        assert np.array_equal(got[offs[1]:offs[1] + len(w)], w)
        assert not got[:offs[1]].any() and not got[offs[1] + len(w):].any()


@pytest.mark.parametrize("elem", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("run", [1, 15, 16, 31, 47, 511, 512, 513, 4095, 4096, 8191, 8193, 65537])
def test_box_copy_rows(elem, run):
    """Rows of about `run` bytes: around the short rows, a row per warp, a
    span per warp and several pieces per row, at every alignment of the two
    sides, rows side by side in dimension 0 or 1, few and many jobs."""
    import torch
    rng = np.random.default_rng(run)
    cols = max(1, run // elem)
    cases = [(1, (1, 1, cols), ((0, 0, 0), (0, 0, 0)), (0, 0)), (1, (1, 9, cols), ((0, 0, 0), (0, 0, 3)), (0, 0)),
             (3, (5, 3, cols), ((0, 1, 2), (1, 0, 5)), (0, 0)), (5, (33, 2, cols), ((2, 0, 0), (0, 2, 7)), (4, 0)),
             (1, (2, 17, cols), ((0, 0, 4), (0, 3, 8)), (0, 4)), (1, (3, 7, cols), ((0, 0, 1), (0, 0, 4)), (1, 6)),
             (44, (1, 2, cols), ((0, 0, 1), (0, 0, 0)), (0, 0)), (45, (2, 1, cols), ((0, 0, 0), (0, 1, 1)), (8, 8))]
    for c in cases:
        _copy_case(torch, rng, *c[:1], elem, *c[1:])
