"""Box copies at the ends of what a job takes: no bytes, and more than its
32-bit row length holds."""
import subprocess
import sys

import numpy as np
import pytest

from paper_2503_10516_gb300 import workloads as W


def test_jobs_without_bytes_copy_nothing():
    """Elements of zero bytes and empty boxes: nothing to copy, not an error
    (in a process of its own: dividing by the row's length ended it)."""
    code = """
from paper_2503_10516_gb300 import igs
jobs = (igs.CopyJob * 2)()
for j, (elem, cols) in zip(jobs, ((0, 3), (4, 0))):
    j.elem_size = elem
    for box in (j.src_box, j.dst_box, j.box):
        box.hi[:] = (1, 2, cols)
assert igs.lib().igs_box_copy(jobs, 2, None) == igs.IGS_OK
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


LONG = (1 << 28) + 5  # 4-byte elements: a row of more than 1 GiB


@pytest.mark.gpu
@pytest.mark.parametrize("ext,src_pad,dst_pad,off", [((1, 1, LONG), 0, 0, 0), ((1, 2, LONG // 2), 0, 0, 1),
                                                     ((1, 2, LONG), 0, 3, 0), ((2, 1, LONG), 1, 0, 2)])
def test_rows_longer_than_a_job(ext, src_pad, dst_pad, off):
    """Contiguous runs of more than 1 GiB: one, rows that form one, and several
    in dimension 1 and 0, at equal and different alignments."""
    import torch
    from paper_2503_10516_gb300 import igs
    planes, rows, cols = ext
    src = torch.empty(planes * rows * (cols + src_pad) + off, dtype=torch.int32, device="cuda")
    torch.arange(src.numel(), out=src)
    dst = torch.full((planes * rows * (cols + dst_pad),), -1, dtype=torch.int32, device="cuda")
    box = lambda pad: (0, 0, 0, planes, rows, cols + pad)  # noqa: E731
    igs.box_copy([(src.data_ptr() + 4 * off, box(src_pad), dst.data_ptr(), box(dst_pad), box(0), 4)],
                 torch.cuda.current_stream().cuda_stream)
    s = src[off:].view(planes, rows, cols + src_pad)[:, :, :cols]
    d = dst.view(planes, rows, cols + dst_pad)
    assert torch.equal(d[:, :, :cols], s)
    assert bool((d[:, :, cols:] == -1).all())


@pytest.mark.gpu
@pytest.mark.parametrize("executor", [0, 1])
def test_buffer_longer_than_a_job(executor):
    """A buffer of more than 1 GiB: uploaded, copied to the device by the
    executor, and read back."""
    from paper_2503_10516_gb300 import igs
    ext = (LONG, 1, 1)
    data = np.arange(LONG, dtype=np.float32)
    c = igs.Context(1, 1, 4, 0, mode=igs.MODE_BATCHED)
    c.set_executor(executor)
    c.create_buffer(1, ext[:1], 4, data)
    c.create_buffer(1, ext[:1], 4, None)
    c.submit(W.Task(1, ext, 1, W.K_SHIFT, [W.Accessor(0, W.READ, W.one_to_one()),
                                           W.Accessor(1, W.WRITE, W.one_to_one())]))
    c.flush()
    c.execute()
    for b in (0, 1):
        got = c.read_buffer(b, (0, 0, 0), ext, 4).view(np.float32).reshape(-1)
        assert np.array_equal(got, data), b
    c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n_jobs", [45, 46, 300])
@pytest.mark.parametrize("order", ["ascending", "descending", "mixed"])
def test_jobs_of_unequal_size(order, n_jobs):
    """Many jobs of 4 bytes to 300 KB (one unit to dozens) in one launch: a
    block finds its job where even sizes would put it, or by search."""
    import torch
    from paper_2503_10516_gb300 import igs
    rng = np.random.default_rng(n_jobs)
    sizes = np.sort(np.exp(rng.uniform(0, np.log(75000), n_jobs)).astype(np.int64))
    if order != "ascending":
        sizes = sizes[::-1] if order == "descending" else rng.permutation(sizes)
    at = np.concatenate([[0], np.cumsum(sizes)])
    src = torch.arange(int(at[-1]), dtype=torch.int32, device="cuda")
    dst = torch.full((int(at[-1]) + 1,), -1, dtype=torch.int32, device="cuda")
    box = [(0, 0, 0, 1, 1, int(s)) for s in sizes]
    igs.box_copy([(src.data_ptr() + 4 * int(a), b, dst.data_ptr() + 4 * int(a) + 4, b, b, 4) for a, b in zip(at, box)],
                 torch.cuda.current_stream().cuda_stream)
    assert torch.equal(dst[1:], src) and int(dst[0]) == -1
