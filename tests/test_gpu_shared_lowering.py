"""Lowering by helper and front warps in the forms that lend them scratch of
the launch (a batch's blocks, the allocation-free entry point), where they and
their staging run out: the graphs are the oracle's all the same."""
import pytest

from paper_2503_10516_gb300 import workloads as W
from tests.harness import assert_same_graph, oracle_graphs
from tests.test_gpu_batch import _stage
from tests.test_zz_no_alloc import _static_graphs

pytestmark = pytest.mark.gpu


def _all_to_all(chunks, nodes, devices, tasks=2, lookahead=0):
    """Every chunk reads every row the others wrote: chunks edges per kernel,
    more of them than the workers' stages hold at 176 chunks. With lookahead
    the rows of a buffer share one allocation per memory."""
    ext = (chunks, 2, 1)
    ops = [("buffer", W.Buffer(2, ext, 4, None, "u32")) for _ in range(2)]
    for k in range(tasks):
        accs = [W.Accessor(k % 2, W.WRITE, W.one_to_one())]
        if k:
            accs.append(W.Accessor((k + 1) % 2, W.READ, W.all_mapper()))
        ops.append(("task", W.Task(2, ext, chunks, W.K_GENERIC, accs)))
    return W.Program(f"all{chunks}x{nodes}x{devices}", nodes, devices, 4, lookahead, ops + [("flush",)])


def _batch_is_the_oracles(progs, ctxs):
    from paper_2503_10516_gb300 import igs
    igs.lower_batch(ctxs)
    for p, c in zip(progs, ctxs):
        ref, rej = oracle_graphs(p)
        assert c.rejected() == rej
        for n in range(p.nodes):
            assert_same_graph(c.graph(n), ref[n], f"{p.name} node {n}")
        c.close()


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("devices", [1, 2])
def test_stages_too_small_for_the_plan(devices, own):
    """200 x 200 edges in 512-entry tables (2048 edges a worker): planned
    kernels fall back to one warp, also where the context has helper scratch of
    its own from an earlier launch."""
    from paper_2503_10516_gb300 import igs
    p = _all_to_all(200, 1, devices)
    c = igs.Context(p.nodes, p.devices, p.horizon_step, p.lookahead, mode=igs.MODE_BATCHED, scratch_capacity=512)
    for op in p.ops:
        if op[0] == "buffer":
            c.create_buffer(op[1].dims, op[1].extent[:op[1].dims], op[1].elem_size, op[1].init)
            if own:
                c.sync()
        elif op[0] == "task":
            c.submit(op[1])
        else:
            c.submit_epoch()
    _batch_is_the_oracles([p], [c])


@pytest.mark.parametrize("tasks", [1, 2, 3, 4, 9])
@pytest.mark.parametrize("nodes,devices", [(1, 1), (1, 4), (3, 1), (4, 2)])
def test_batch_pool_shapes(nodes, devices, tasks):
    """Few and many items (a front warp from four on), one and several
    devices, programs of different capacities in one launch, lowered in two
    parts."""
    from paper_2503_10516_gb300 import igs
    progs = [_all_to_all(nodes * devices * 3, nodes, devices, tasks, lookahead=2),
             W.wave_program(n=48, steps=tasks, nodes=nodes, devices=devices, chunks=nodes * devices * 2),
             W.growing_program(rows_max=60, cols=3, devices=2, chunks=2, lookahead=tasks, seed=tasks)]
    ctxs = [_stage(p, igs.MODE_BATCHED) for p in progs]
    igs.lower_batch(ctxs[1:])
    _batch_is_the_oracles(progs, ctxs)


def test_batch_of_equal_programs_keeps_one_warp():
    """Units of equal length past twice the SMs: one warp each, as before."""
    from paper_2503_10516_gb300 import igs
    progs = [W.wave_program(n=32, steps=3, nodes=4, devices=2, chunks=8, seed=i) for i in range(80)]
    ctxs = [_stage(p, igs.MODE_BATCHED) for p in progs]
    _batch_is_the_oracles(progs[:1], ctxs[:1])
    igs.lower_batch(ctxs[1:])
    ref, _ = oracle_graphs(progs[0])
    for c in ctxs[1:]:
        for n in range(4):
            assert_same_graph(c.graph(n), ref[n], f"node {n}")
        c.close()


@pytest.mark.parametrize("prog", [_all_to_all(176, 1, 1, 3, lookahead=4), _all_to_all(176, 1, 4, 3, lookahead=4),
                                  _all_to_all(24, 8, 1, 5),
                                  W.wave_program(n=40, steps=6, nodes=9, devices=2, chunks=18),
                                  W.wave_program(n=40, steps=2, nodes=8, devices=3, chunks=24, lookahead=4)],
                         ids=lambda p: p.name)
def test_static_shared(prog):
    """Plans that overflow (lowered again by one warp), one device per node,
    the most nodes that are helped and one more, few items."""
    ref, rej = oracle_graphs(prog)
    assert not rej
    got = _static_graphs(prog)
    for n in range(prog.nodes):
        assert_same_graph(got[n], ref[n], f"{prog.name} node {n}")
