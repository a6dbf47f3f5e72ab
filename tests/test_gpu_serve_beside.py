"""Calls made while a serving loop holds the device: none waits for the loop to
end, although each is the process's first use of its kernels."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes, time
import torch
from paper_2503_10516_gb300 import igs, workloads as W

def context(prog):
    c = igs.Context(prog.nodes, prog.devices, prog.horizon_step, prog.lookahead, mode=igs.MODE_BATCHED,
                    max_instructions=20000, map_heap=1 << 16)
    for b in prog.buffers:
        c.create_buffer(b.dims, b.extent[:b.dims], b.elem_size, b.init)
    return c

def submitted(**shape):
    prog = W.jacobi_program(n=64, lookahead=0, nodes=1, **shape)
    c = context(prog)
    for t in prog.tasks:
        c.submit(t)
    return c

def copies(n):
    jobs = (igs.CopyJob * n)()
    for j in range(n):
        jobs[j].src, jobs[j].dst, jobs[j].elem_size = mem.data_ptr(), mem.data_ptr() + (j + 1) * 64, 4
        for box in (jobs[j].src_box, jobs[j].dst_box, jobs[j].box):
            box.hi[:] = (1, 1, 16)
    assert igs.lib().igs_box_copy(jobs, n, stream.cuda_stream) == igs.IGS_OK

mem = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda")
stream = torch.cuda.Stream()
few, many = dict(steps=4, devices=2, chunks=4), dict(steps=40, devices=4, chunks=16)
one = submitted(steps=4, devices=1, chunks=4)
ctxs = [submitted(**few), submitted(**many), submitted(**few)]
prog = W.growing_program(rows_max=64, cols=4, nodes=1, devices=2, chunks=2, lookahead=0, seed=1)
served = context(prog)
server = igs.Server(max_slots=4, idle_timeout_ms=2000)
assert server.attach(served, 256) == igs.IGS_OK
torch.cuda.synchronize()
server.start()
time.sleep(0.1)
calls = [("copies of 1", lambda: copies(1)), ("copies of 10", lambda: copies(10)), ("copies of 40", lambda: copies(40)),
         ("flush, one device", one.flush), ("batch, one warp", lambda: igs.lower_batch(ctxs[:1])),
         ("batch, lent warps", lambda: igs.lower_batch(ctxs[1:2])),
         ("batch, work queue", lambda: igs.lower_batch(ctxs[2:], (4, 1)))]
for name, call in calls:
    t = time.perf_counter()
    call()
    t = time.perf_counter() - t
    assert t < 1.0, f"{name}: {t:.2f} s"
assert ctxs[0].profile()["n_shared_phases"] == 0 < ctxs[1].profile()["n_shared_phases"]
server.stop()
"""


def test_first_calls_beside_the_loop():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
