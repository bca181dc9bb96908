"""Barrier-free sweep by trip maps (csrc/trip.cuh) against the oracle, at the
sizes where they can go wrong: trips around the shortest it takes and the 32
iterations of a batch, bodies up to 32 records, offsets up to the farthest a
map carries and past it, waits on outer loops' producers, more inputs than a
map holds, and thresholds that name other increments, which the walk takes."""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import ALL_MODES, compare_all

pytestmark = pytest.mark.gpu

PRM = dict(ii=2, c_branch=3, c_regop=2)


@pytest.fixture(scope="module")
def sg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13757_gb300 import build
    build.build()
    import paper_2608_13757_gb300 as m
    return m


def program(trips, records, engines, density, k_max, rng):
    """Leaf loop of `records` instructions inside a loop, its waits carried at
    offsets 0..k_max, from and to the loop around it."""
    b = workloads.ProgramBuilder(engines)
    eng = lambda: int(rng.integers(0, engines))
    lat = lambda: int(rng.integers(1, 200))
    A = b.loop(0, 0, [len(trips)])
    a0, a1 = b.instr(A, 0, eng(), lat()), b.instr(A, 1, eng(), lat())
    L = b.loop(A, 2, trips)
    xs = [b.instr(L, i, eng(), lat()) for i in range(records)]
    a2 = b.instr(A, 3, eng(), lat())
    for i in range(records):
        if i and rng.random() < density:
            b.dep(xs[int(rng.integers(0, i))], xs[i], 0)
        if rng.random() < density:
            b.dep(xs[int(rng.integers(0, records))], xs[i], int(rng.integers(1, k_max + 1)))
        if rng.random() < density / 3:
            b.dep((a0, a1)[i & 1], xs[i], 0)
    b.dep(xs[-1], a2, 0)
    b.dep(xs[0], a0, 1)
    b.dep(a2, xs[0], 1)
    return b.batch()


def fixed_program(trips, records, rng):
    """A loop of conditionals taken always, some nested, beside records of its
    own, each instruction waiting for the one before it, and a record no
    engine of the body runs."""
    b = workloads.ProgramBuilder(5)
    A = b.loop(0, 0, [len(trips)])
    L = b.loop(A, 0, trips)
    n = sum(trips)
    xs, where = [], L
    for i in range(records):
        where = b.loop(L, i, [1] * n) if i % 3 else L
        if i % 3 == 2:
            where = b.loop(where, 0, [1] * n)
        xs.append(b.instr(where, i, int(rng.integers(0, 4)), int(rng.integers(1, 200))))
    z = b.instr(A, 1, 4, 7)
    for p, c in zip(xs, xs[1:]):
        b.dep(p, c, 0)
    b.dep(xs[-1], xs[0], 1)
    b.dep(xs[3 * ((records - 1) // 3)], xs[0], 2)
    b.dep(xs[-1], xs[-1], 1)
    b.dep(xs[-1], z, 0)
    b.dep(z, xs[0], 1)
    return b.batch()


def batch_of(rng):
    trips = [[40] + [t, t + 1, 0, 64, t] for t in (1, 3, 4, 31, 32, 33, 65)]
    shapes = [(1, 1, 0.9, 1), (2, 2, 0.9, 3), (5, 3, 0.6, 4), (16, 4, 0.4, 2), (17, 5, 0.3, 3), (32, 8, 0.15, 2),
              (32, 2, 0.8, 2), (31, 12, 0.2, 1)]
    return workloads.concat([program(t, *s, rng) for t in trips for s in shapes] +
                            [fixed_program(t, n, rng) for t in trips for n in (1, 2, 7, 20)])


@pytest.mark.parametrize("seed", range(2))
def test_trip_edges(sg, seed):
    batch = batch_of(np.random.default_rng(seed))
    compare_all(sg, batch, timeline=True, modes=ALL_MODES, params=oracle.sim_params(**PRM))


def test_trip_costs(sg):
    batch = batch_of(np.random.default_rng(5))
    compare_all(sg, batch, timeline=True, modes=ALL_MODES,
                params=oracle.sim_params(licm=1, cse=1, trip_register_elision=1, **PRM))


@pytest.mark.parametrize("mode", [oracle.COUNT, oracle.PERLOOP])
def test_waits_on_other_increments(sg, mode):
    """Thresholds moved to earlier increments, to none and past the end."""
    import torch
    rng = np.random.default_rng(9)
    batch = workloads.concat([program([40, 50, 33, 70], 16, 4, 0.4, 2, rng) for _ in range(16)])
    h = sg.sync_load_programs(batch)
    want = oracle.thresholds(batch, mode).copy()
    own = np.repeat(np.arange(batch.n_deps), h.pair_counts)
    prog = np.searchsorted(batch.prog_dep_ptr, own, side="right") - 1
    for p in range(15):
        at = rng.choice(np.flatnonzero((prog == p) & (want > 0)))
        want[at] = max(0, want[at] + (-1, -9, -want[at], 10 ** 6, 1)[p % 5])
    thr = sg.sync_eval_thresholds(h, mode)
    thr[torch.from_numpy(h.unpadded_index()).to(thr.device)] = torch.from_numpy(want).to(thr.device)
    ref = oracle.simulate(batch, want, mode, oracle.BARRIER_FREE)
    r = sg.sync_simulate(h, mode, thr)
    P = batch.n_programs
    assert np.array_equal(r.status.cpu().numpy()[:P], ref.status)
    assert np.array_equal(r.makespan.cpu().numpy()[:P], ref.makespan)
    assert np.array_equal(r.checksum.cpu().numpy()[:P].view(np.uint64), ref.checksum)
    assert (ref.status == 0).any() and (ref.status != 0).any()
    h.close()


@pytest.mark.parametrize("config", ["syncbound", "small"])
@pytest.mark.parametrize("programs", [1, 7, 151, 152, 153, 305, 1216, 1217, 1368, 2433, 3649])
def test_programs_over_the_sms(sg, config, programs):
    """Batches around a warp, 8 warps and whole CTAs on every SM, whose
    sweeps take CTAs of 1 to 8 warps."""
    compare_all(sg, workloads.generate(config, n_programs=programs), modes=[oracle.PERLOOP])


def many_waits(waited, reps, rng):
    """A loop of `reps` iterations around `waited` producers, each waited on
    by a consumer of its own, beside a leaf loop of long trips."""
    b = workloads.ProgramBuilder(4)
    A = b.loop(0, 0, [reps])
    for i in range(waited - 1):
        p = b.instr(A, 2 * i, i % 3, int(rng.integers(1, 50)))
        b.dep(p, b.instr(A, 2 * i + 1, 3, 2), 0)
    L = b.loop(A, 2 * waited, [64] * reps)
    xs = [b.instr(L, i, i % 2, int(rng.integers(1, 50))) for i in range(9)]
    b.dep(xs[0], xs[1], 0)
    return b.batch()


@pytest.mark.parametrize("waited", [24, 28, 32, 239, 240, 241, 244, 245, 320, 321, 440])
def test_many_waited_semaphores(sg, waited):
    """Rings of fewer increments, maps on fewer CTAs, and numbers of
    semaphores that leave no ring beside the maps, in batches whose sweep
    takes maps otherwise; also through the call that allocates nothing."""
    import torch
    rng = np.random.default_rng(waited)
    batch = workloads.concat([many_waits(waited, 20, rng)] + [program([70] * 40, 17, 5, 0.3, 2, rng) for _ in range(8)])
    h = compare_all(sg, batch, modes=[oracle.COUNT])
    thr = sg.sync_eval_thresholds(h, oracle.COUNT)
    want, got = sg.sync_simulate(h, oracle.COUNT, thr), sg.sync_simulate_noalloc(h, oracle.COUNT, thr)
    for f in ("status", "makespan", "checksum"):
        assert torch.equal(getattr(got, f), getattr(want, f))


def test_too_many_waited_semaphores(sg):
    h = sg.sync_load_programs(many_waits(460, 20, np.random.default_rng(1)))
    thr = sg.sync_eval_thresholds(h, oracle.COUNT)
    for call in (sg.sync_simulate, sg.sync_simulate_noalloc):
        with pytest.raises(sg.SyncError) as err:
            call(h, oracle.COUNT, thr)
        assert err.value.status == sg.ERR_ARG
