"""Stencil tasks whose ranges do not match the buffers they read, or one another."""
import numpy as np
import pytest

from paper_2503_10516_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("executor", [0, 1])
@pytest.mark.parametrize("chunks", [1, 3])
@pytest.mark.parametrize("kind", ["jacobi", "wave"])
@pytest.mark.parametrize("read", [(8, 16), (16, 8), (5, 7)], ids=str)
def test_range_larger_than_the_buffer_it_reads(read, kind, chunks, executor):
    """Items outside the buffer they read are reported and see zeros; the
    others compute what they would alone."""
    from paper_2503_10516_gb300 import igs
    n = 16
    rng = np.random.default_rng(1)
    u, prev = rng.random(read, dtype=np.float32), rng.random((n, n), dtype=np.float32)
    c = igs.Context(1, 2, 4, 0, mode=igs.MODE_BATCHED)
    c.set_executor(executor)
    c.create_buffer(2, read, 4, u)
    c.create_buffer(2, (n, n), 4, prev)
    c.create_buffer(2, (n, n), 4, None)
    accs = [W.Accessor(0, W.READ, W.neighborhood(1, 1)), W.Accessor(2, W.WRITE, W.one_to_one())]
    if kind == "wave":
        accs.insert(0, W.Accessor(1, W.READ, W.one_to_one()))
    c.submit(W.Task(2, (n, n, 1), chunks, W.K_WAVE if kind == "wave" else W.K_JACOBI, accs))
    c.flush()
    with pytest.raises(igs.IgsError) as e:
        c.execute()
    assert e.value.code == igs.IGS_ERR_OUT_OF_BOUNDS
    want = np.zeros((n, n), np.float32)
    want[:read[0], :read[1]] = u
    inner = (slice(1, read[0] - 1), slice(1, read[1] - 1))
    cen, t5 = u[1:-1, 1:-1], (u[:-2, 1:-1] + u[2:, 1:-1]) + (u[1:-1, :-2] + u[1:-1, 2:])
    if kind == "jacobi":
        want[inner] = t5 * np.float32(0.25)
    else:
        want[inner] = (np.float32(2) * cen - prev[inner]) + np.float32(0.25) * (t5 - np.float32(4) * cen)
    got = c.read_buffer(2, (0, 0, 0), (n, n, 1), 4).view(np.float32).reshape(n, n)
    c.close()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("devices", [1, 2])
@pytest.mark.parametrize("thin", [((40, 33), 20), ((3, 700), 3), ((1, 5), 1), ((130, 64), 65)], ids=str)
def test_jobs_of_unequal_size_in_one_level(thin, devices):
    """Two independent sweeps that share their levels: few large chunks, and
    many (or as many) small ones, whose tiles are found by search."""
    from paper_2503_10516_gb300 import igs
    rng = np.random.default_rng(3)
    sweeps = [((150, 300), 2)] + [thin]
    c = igs.Context(1, devices, 4, 0, mode=igs.MODE_BATCHED)
    init = [rng.random(shape, dtype=np.float32) for shape, _ in sweeps]
    for (shape, _), u in zip(sweeps, init):
        c.create_buffer(2, shape, 4, u)
        c.create_buffer(2, shape, 4, None)
    steps = 3
    for k in range(steps):
        for i, (shape, chunks) in enumerate(sweeps):
            c.submit(W.Task(2, (*shape, 1), chunks, W.K_JACOBI, [
                W.Accessor(2 * i + k % 2, W.READ, W.neighborhood(1, 1)),
                W.Accessor(2 * i + (k + 1) % 2, W.WRITE, W.one_to_one())]))
    c.flush()
    c.execute()
    for i, ((shape, _), u) in enumerate(zip(sweeps, init)):
        for _ in range(steps):
            out = u.copy()
            out[1:-1, 1:-1] = ((u[:-2, 1:-1] + u[2:, 1:-1]) + (u[1:-1, :-2] + u[1:-1, 2:])) * np.float32(0.25)
            u = out
        got = c.read_buffer(2 * i + steps % 2, (0, 0, 0), (*shape, 1), 4).view(np.float32).reshape(shape)
        assert np.array_equal(got, u), shape
    c.close()
