"""Batches at the edge of a context's capacities: a launch that lends its
blocks' helper and front warps to the nodes answers as one warp per node does,
whatever runs out where."""
import pytest

from paper_2503_10516_gb300 import workloads as W
from tests.harness import assert_same_graph, oracle_graphs

pytestmark = pytest.mark.gpu


def _context(prog, **caps):
    from paper_2503_10516_gb300 import igs
    return igs.Context(prog.nodes, prog.devices, prog.horizon_step, prog.lookahead, mode=igs.MODE_BATCHED,
                       max_instructions=8192, max_edges=1 << 18, max_boxes=1 << 15, max_queue=256, **caps)


def _submit(c, ops):
    for op in ops:
        if op[0] == "buffer":
            c.create_buffer(op[1].dims, op[1].extent[:op[1].dims], op[1].elem_size, op[1].init)
        elif op[0] == "task":
            c.submit(op[1])
        elif op[0] == "destroy":
            c.destroy_buffer(op[1])
        else:
            c.submit_epoch()


def _lower(prog, parts, shape, **caps):
    """The program's graphs, lowered by one batch per part of its operations;
    None where a capacity ran out."""
    from paper_2503_10516_gb300 import igs
    c = _context(prog, **caps)
    try:
        for ops in parts:
            _submit(c, ops)
            igs.lower_batch([c], shape)
        return [c.graph(n) for n in range(prog.nodes)]
    except igs.IgsError as e:
        assert e.code == igs.IGS_ERR_CAPACITY
        return None
    finally:
        c.close()


def _pieces_program():
    """170 rows written on two devices. The kernels of the second task read
    the inner columns of all rows: their edges (170 each) overflow the workers'
    stages (1024 edges at 256 entries), while the up-to-date bits of the
    copies, set beside that plan, split the rows' state into pieces. The last
    task reads one such row whole, so it copies what the bits say."""
    ext = (170, 4, 1)
    ops = [("buffer", W.Buffer(2, ext, 4, None, "u32"))]
    ops.append(("task", W.Task(2, ext, 170, W.K_NOP, [W.Accessor(0, W.WRITE, W.one_to_one())])))
    for chunks, box in ((48, W.fixed_box((0, 1), (170, 3))), (2, W.fixed_box((84, 0), (85, 4)))):
        ops.append(("task", W.Task(2, ext, chunks, W.K_NOP, [W.Accessor(0, W.READ, box)])))
    return W.Program("pieces", 1, 2, 100, 1, ops)


def test_state_table_runs_out_beside_an_overflowing_plan():
    """Whichever table the heap runs out for while the kernel plan overflows
    its stages: the lowering ends with a capacity error or is the oracle's."""
    prog = _pieces_program()
    ref, _ = oracle_graphs(prog)
    done = []
    for heap in range(2048, 4352, 64):
        got = _lower(prog, [prog.ops], None, map_heap=heap, scratch_capacity=256)
        if got is not None:
            done.append(heap)
            assert_same_graph(got[0], ref[0], f"heap of {heap} entries")
    assert done and done[0] > 2048  # the range reaches from too small to enough


def _rotating_program(nodes, devices, steps):
    """A new buffer per task, read transposed by the next task and then
    destroyed: ownership and state tables come and go."""
    ext = (16, 16, 1)
    ops = []
    for k in range(steps):
        ops.append(("buffer", W.Buffer(2, ext, 4, None, "u32")))
        accs = [W.Accessor(k, W.WRITE, W.one_to_one())]
        if k:
            accs.append(W.Accessor(k - 1, W.READ, W.transposed()))
        ops.append(("task", W.Task(2, ext, 16, W.K_NOP, accs)))
        if k > 1:
            ops.append(("destroy", k - 2))
    return W.Program(f"rotate{nodes}x{devices}", nodes, devices, 4, 0, ops + [("flush",)])


ALONE = (0, 0)  # igs_lower_batch_shaped: one warp per node


@pytest.mark.parametrize("parts", [1, 2])
@pytest.mark.parametrize("nodes,devices", [(1, 4), (4, 1), (4, 2)])
def test_heap_that_suffices_for_one_warp(nodes, devices, parts):
    """Helper and front warps take slabs in another order than one warp: where
    that exhausts a heap that one warp gets by with, in a context's first launch
    or in a later one, the graph is the oracle's all the same."""
    prog = _rotating_program(nodes, devices, 12)
    ref, _ = oracle_graphs(prog)
    cut = len(prog.ops) // 2
    pieces = [prog.ops[:cut], prog.ops[cut:]] if parts == 2 else [prog.ops]

    def lower(heap, shape):
        return _lower(prog, pieces, shape, map_heap=heap, scratch_capacity=1024)
    too_small, least = 128, 8192
    assert lower(too_small, ALONE) is None and lower(least, ALONE) is not None
    while least - too_small > 32:
        mid = (too_small + least) // 64 * 32
        if lower(mid, ALONE) is None:
            too_small = mid
        else:
            least = mid
    assert lower(too_small, None) is None
    for heap in range(least, least + 512, 32):
        got = lower(heap, None)
        assert got is not None, f"a heap of {least} entries suffices for one warp, {heap} do not"
        for n in range(nodes):
            assert_same_graph(got[n], ref[n], f"node {n}, heap of {heap} entries")


@pytest.mark.parametrize("nodes,devices,chunks,tasks,lent", [
    (1, 1, 2, 1, False), (1, 1, 2, 4, False), (4, 2, 16, 1, False), (1, 2, 96, 1, True), (1, 2, 96, 2, True),
    (1, 1, 96, 3, True), (4, 2, 16, 24, True), (1, 4, 16, 9, True)])
def test_form_of_a_batch(nodes, devices, chunks, tasks, lent):
    """Warps are lent where there is enough to lower, also for one, two and
    three items; small calls keep one warp per node. Lowered twice, so that the
    second call is not the context's first."""
    from paper_2503_10516_gb300 import igs
    ext = (max(chunks, 8), 8, 1)
    ops = [("buffer", W.Buffer(2, ext, 4, None, "u32")) for _ in range(2)]
    for k in range(tasks):
        accs = [W.Accessor(k % 2, W.WRITE, W.one_to_one())]
        if k:
            accs.append(W.Accessor((k + 1) % 2, W.READ, W.neighborhood(1)))
        ops.append(("task", W.Task(2, ext, chunks, W.K_NOP, accs)))
    prog = W.Program("form", nodes, devices, 4, 0, ops + ops[2:])
    ref, _ = oracle_graphs(prog)
    c = igs.Context(nodes, devices, 4, 0, mode=igs.MODE_BATCHED)
    phases = [0]
    for part in (ops, ops[2:]):
        _submit(c, part)
        igs.lower_batch([c])
        phases.append(c.profile()["n_shared_phases"])
        assert (phases[-1] > phases[-2]) == lent
    for n in range(nodes):
        assert_same_graph(c.graph(n), ref[n], f"node {n}")
    c.close()


@pytest.mark.parametrize("devices", [2, 3])
def test_coherence_plan_overflows(devices):
    """Every copy of the fourth task overwrites rows that up to 100 kernels of
    the second read: some 10^4 edges for the one or two workers that plan a
    memory, 2048 in a stage. The phase is taken by one warp, then the kernels."""
    from paper_2503_10516_gb300 import igs
    ext = (200, 2, 1)
    ops = [("buffer", W.Buffer(2, ext, 4, None, "u32")) for _ in range(2)]
    for k in range(4):
        accs = [W.Accessor(k % 2, W.WRITE, W.one_to_one())]
        if k:
            accs.append(W.Accessor((k + 1) % 2, W.READ, W.all_mapper()))
        ops.append(("task", W.Task(2, ext, 200, W.K_NOP, accs)))
    prog = W.Program("overwrite", 1, devices, 100, 2, ops + [("flush",)])
    ref, _ = oracle_graphs(prog)
    c = igs.Context(1, devices, 100, 2, mode=igs.MODE_BATCHED, scratch_capacity=512)
    _submit(c, prog.ops)
    igs.lower_batch([c])
    assert c.profile()["n_shared_phases"] > 0
    assert_same_graph(c.graph(0), ref[0])
    c.close()
