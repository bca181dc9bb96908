"""Which barrier-free batches take trips by their maps (sweep_maps in
csrc/k_sweep.cu), on the host: only those whose loops a map can take for most
of their work -- trips that follow each other, of bodies up to 32 records,
after the iterations walked first -- and whose gain outweighs the fewer warps.
And which programs the barrier scheme takes by intervals: those whose walk is
longer than laying them out."""
import ctypes

import numpy as np
import pytest

import paper_2608_13757_gb300 as sg
import workloads

SMS = 152


def takes_maps(batch, waited=4):
    desc, keep = sg.batch_desc(batch)
    got = sg.lib().syncgb_takes_maps(ctypes.byref(desc), SMS, waited)
    assert got in (0, 1) and keep
    return bool(got)


def leaves(records, trip, visits, n_leaves, inner=0, nested=False):
    """A loop of `visits` iterations around `n_leaves` leaf loops of `trip`
    iterations each; `inner`: that many of the records in loops that run once
    on every visit; nested: the loop around them is itself in one."""
    b = workloads.ProgramBuilder(4)
    A = b.loop(0, 0, [1]) if nested else 0
    A = b.loop(A, 0, [visits])
    for q in range(n_leaves):
        L = b.loop(A, q, [trip] * visits)
        xs = [b.instr(b.loop(L, i, [1] * (trip * visits)) if i < inner else L, i, i % 4, 10 + i) for i in range(records)]
        for i in range(1, records, 2):
            b.dep(xs[i - 1], xs[i], 0)
        b.dep(xs[-1], xs[0], 1)
    return b.batch()


def many(one, n):
    out, have = None, one
    while n:
        if n & 1:
            out = have if out is None else workloads.concat([out, have])
        have = workloads.concat([have, have]) if n > 1 else have
        n >>= 1
    return out


@pytest.mark.parametrize("programs", [1, 1000, 2500, 3500, 5000, 12000])
def test_loops_entered_once_are_walked(programs):
    assert not takes_maps(workloads.generate("small", n_programs=programs))


@pytest.mark.parametrize("programs", [1, 500, 3000])
@pytest.mark.parametrize("shape,maps", [
    ((16, 64, 16, 1), True),              # trips a map takes
    ((32, 32, 32, 1), True),
    ((33, 64, 16, 1), False),             # more records than lanes
    ((40, 64, 64, 1), False),
    ((16, 64, 64, 2), False),             # two loops in turn: the warp keeps one map
    ((16, 64, 1, 1), False),              # entered once: walked while it is learned
    ((16, 3, 300, 1), False),             # trips too short for a map
    ((16, 64, 16, 1, 5), True),           # around loops that run once
    ((16, 64, 16, 1, 0, True), True)])
def test_shapes(shape, maps, programs):
    assert takes_maps(many(leaves(*shape), programs)) == maps


def test_few_trips_of_many_programs():
    assert takes_maps(many(leaves(16, 64, 4, 1), 12000)) and takes_maps(many(leaves(16, 16, 64, 1), 6000))


def test_short_work_needs_the_warps():
    """Trips of 8: by maps while every warp has few neighbours, walked where
    24 warps an SM take the batch at once and 16 do not."""
    one = leaves(16, 8, 128, 1)
    assert takes_maps(many(one, 500)) and not takes_maps(many(one, 3000)) and not takes_maps(many(one, 20000))
    assert not takes_maps(many(leaves(4, 32, 32, 1), 3000))


@pytest.mark.parametrize("config,programs,maps", [
    ("chain", 300, True), ("chain", 4096, True), ("chain", 12000, True), ("chain", 32768, False),
    ("depth2", 1500, True), ("depth2", 16384, True), ("syncbound", 777, True), ("syncbound", 20000, True),
    ("attention", 2, True), ("gemm", 1, False)])
def test_configurations(config, programs, maps):
    assert takes_maps(workloads.generate(config, n_programs=programs)) == maps


def test_waits_inside_a_chunk_make_the_walk_longer():
    """A body without waits inside an iteration is walked in one pass a chunk:
    the same loop in many programs stays with the walk."""
    b = workloads.ProgramBuilder(5)
    A = b.loop(0, 0, [18])
    L = b.loop(A, 0, [6, 7, 7, 8, 9, 11, 13, 18, 18, 21, 24, 25, 26, 27, 28, 30, 31, 32])
    xs = [b.instr(L, i, i % 5, 10 + i) for i in range(12)]
    for i in range(3):
        b.dep(xs[i], xs[i + 4], 2)
    apart = b.batch()
    for i in range(1, 12, 2):
        b.dep(xs[i - 1], xs[i], 0)
    assert takes_maps(apart) and not takes_maps(many(apart, 3000))
    assert takes_maps(b.batch()) and takes_maps(many(b.batch(), 3000))


@pytest.mark.parametrize("shape", [(8, 16, 4, 1), (4, 16, 16, 1), (4, 64, 4, 1)])
def test_building_the_map_has_to_pay(shape):
    assert not takes_maps(leaves(*shape)) and not takes_maps(many(leaves(*shape), 1000))


def test_waited_semaphores():
    """Rings that leave the maps one CTA per SM and the walk three, two and
    one, and no ring beside the maps."""
    batch = many(leaves(16, 16, 64, 1), 3000)
    assert [takes_maps(batch, n) for n in (4, 28, 36, 120, 240, 241)] == [True, True, False, True, True, False]


def test_loops_with_fallback_barriers_are_walked():
    from tests.test_fallback_pins import with_policy
    b = workloads.ProgramBuilder(2)
    A = b.loop(0, 0, [16])
    S = b.loop(A, 0, [64] * 16)
    p = b.instr(b.loop(S, 0, [1] * 1024), 0, 0, 50)
    c = b.instr(S, 1, 1, 3)
    assert takes_maps(b.batch())
    b.dep(p, c, 2)
    assert not takes_maps(with_policy(b.batch(), 1))


def test_divergent_batches_are_walked():
    assert not takes_maps(workloads.diverge(workloads.generate("depth2", n_programs=40), 5, permille=300))


def test_batches_of_the_other_tests_take_maps():
    """The batches with which the maps themselves are tested."""
    from tests import test_gpu_trips as t
    from tests.test_fallback_pins import with_policy
    from tests.test_gpu_fallback import flagged_program
    rng = np.random.default_rng(0)
    assert takes_maps(t.batch_of(rng))
    assert takes_maps(workloads.concat([t.program([40, 50, 33, 70], 16, 4, 0.4, 2, rng) for _ in range(16)]))
    assert takes_maps(workloads.concat([t.many_waits(440, 20, rng)] +
                                       [t.program([70] * 40, 17, 5, 0.3, 2, rng) for _ in range(8)]), 240)
    assert takes_maps(with_policy(workloads.concat([flagged_program("host", False)] +
                                                   [t.fixed_program([64] * 40, 7, rng) for _ in range(12)]), 1))


def test_refused_batch():
    b = workloads.generate("small").copy()
    b.instr_latency[:] = 0
    desc, keep = sg.batch_desc(b)
    assert sg.lib().syncgb_takes_maps(ctypes.byref(desc), SMS, 4) == -1 and keep


@pytest.mark.parametrize("shape,few,many_", [
    ((16, 64, 1, 1), False, False),       # one trip: its iterations replay
    ((24, 16, 4, 1), False, False),
    ((8, 16, 2, 2), False, False),        # sibling loops
    ((16, 64, 16, 1), True, True),
    ((2, 4, 32, 1), True, True),          # short trips
    ((40, 32, 4, 1), True, True),         # more records than lanes
    ((5, 16, 8, 1, 5), True, True)])      # conditionals around one record
def test_programs_by_intervals(shape, few, many_):
    desc, keep = sg.batch_desc(leaves(*shape))
    got = sg.lib().syncgb_by_intervals(ctypes.byref(desc))
    assert keep and (got & 1, got & 2) == (1 if few else 0, 2 if many_ else 0)
    assert not got & 3 or got >> 2 & got & 3 == got & 3
