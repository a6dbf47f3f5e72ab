"""Box-copy jobs as the host splits them, as far as no GPU is needed."""
import subprocess
import sys


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
