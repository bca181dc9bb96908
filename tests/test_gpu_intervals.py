"""Barrier scheme by intervals (csrc/bar.cuh) against the oracle, at the sizes
where its tiles and row searches can go wrong: trip totals around a lane, a
warp and a tile, rows without iterations, bodies of more records than lanes,
loops that run exactly once, moving loops beside each other, and thresholds
that do not repeat, which send the program to the walk."""
import numpy as np
import pytest

import oracle
import workloads
from tests.test_gpu_parity import ALL_MODES, compare_all

pytestmark = pytest.mark.gpu

PRM = dict(ii=2, c_branch=3, c_regop=2, c_barrier=9)


@pytest.fixture(scope="module")
def sg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13757_gb300 import build
    build.build()
    import paper_2608_13757_gb300 as m
    return m


@pytest.fixture(autouse=True)
def every_program_by_intervals(monkeypatch):
    """The shapes here are small: by default most would be walked."""
    monkeypatch.setenv("SYNCGB_INTERVALS", "1")


def trips_of(total, rows, empty, rng):
    """`rows` trips that add up to `total`, a share `empty` of them 0."""
    t = np.zeros(rows, dtype=np.int64)
    live = np.flatnonzero(rng.random(rows) >= empty)
    if live.size == 0:
        live = np.array([rows - 1])
    np.add.at(t, rng.choice(live, size=total), 1)
    return t.tolist()


def program(total, rows, records, empty, rng):
    """An outer loop of `rows` iterations around a leaf of `total`, with a
    conditional taken always, one taken at times and a second moving loop."""
    b = workloads.ProgramBuilder(3)
    lat = lambda: int(rng.integers(1, 40))
    A = b.loop(0, 1, [rows])
    first = b.instr(0, 0, 0, lat())
    a0 = b.instr(A, 0, 1, lat())
    L = b.loop(A, 1, trips_of(total, rows, empty, rng))
    once = b.loop(A, 2, [1] * rows)
    inner = b.loop(once, 1, [1] * rows)
    x0, x1, x2 = b.instr(once, 0, 2, lat()), b.instr(inner, 0, 0, lat()), b.instr(once, 2, 1, lat())
    M = b.loop(A, 3, rng.integers(0, 3, size=rows).tolist())
    c = b.loop(A, 4, rng.integers(0, 2, size=rows).tolist())
    y, z, w = b.instr(M, 0, 2, lat()), b.instr(c, 0, 0, lat()), b.instr(A, 5, 1, lat())
    xs = [b.instr(L, i, int(rng.integers(0, 3)), lat()) for i in range(records)]
    for i in range(1, records):
        if rng.random() < 0.5:
            b.dep(xs[int(rng.integers(0, i))], xs[i], 0)
        if rng.random() < 0.3:
            b.dep(xs[int(rng.integers(i, records))], xs[i], 1 + int(rng.integers(0, 2)))
    for p, q, k in ((first, xs[0], 0), (a0, xs[-1], 0), (x0, x1, 0), (x1, x2, 0), (x2, x0, 1), (xs[0], x1, 0),
                    (x1, y, 0), (y, z, 0), (z, w, 0), (w, a0, 1), (xs[-1], a0, 1), (y, xs[0], 1)):
        b.dep(p, q, k)
    return b.batch()


@pytest.mark.parametrize("rows,empty", [(1, 0.0), (5, 0.0), (90, 0.6)])
def test_tile_edges(sg, rows, empty):
    rng = np.random.default_rng(rows)
    parts = [program(total, rows, records, empty, rng)
             for total in (0, 1, 31, 32, 33, 127, 128, 129, 385, 513) for records in (1, 3, 17, 33, 66)]
    compare_all(sg, workloads.concat(parts), timeline=True, modes=ALL_MODES, params=oracle.sim_params(**PRM))


@pytest.mark.parametrize("mode", [oracle.COUNT, oracle.PERLOOP])
def test_waits_that_do_not_repeat(sg, mode):
    """Single thresholds moved to earlier increments, to none and past the
    end: the walk's results, deadlocks among them."""
    import torch
    rng = np.random.default_rng(11)
    batch = workloads.concat([program(129, 7, 9, 0.2, rng) for _ in range(12)])
    h = sg.sync_load_programs(batch)
    want = oracle.thresholds(batch, mode).copy()
    own = np.repeat(np.arange(batch.n_deps), h.pair_counts)
    prog = np.searchsorted(batch.prog_dep_ptr, own, side="right") - 1
    for p in range(0, 11):
        at = np.flatnonzero((prog == p) & (want > 0))
        want[rng.choice(at)] += (-1, 1, -want[at].max(), 10 ** 6)[p % 4] if p < 8 else 0
    want = np.maximum(want, 0)
    thr = sg.sync_eval_thresholds(h, mode)
    thr[torch.from_numpy(h.unpadded_index()).to(thr.device)] = torch.from_numpy(want).to(thr.device)
    ref = oracle.simulate(batch, want, mode, oracle.BARRIER)
    r = sg.sync_simulate(h, mode, thr, variant=oracle.BARRIER)
    P = batch.n_programs
    assert np.array_equal(r.status.cpu().numpy()[:P], ref.status)
    assert np.array_equal(r.makespan.cpu().numpy()[:P], ref.makespan)
    assert np.array_equal(r.checksum.cpu().numpy()[:P].view(np.uint64), ref.checksum)
    assert (ref.status == 0).any() and (ref.status != 0).any()
    h.close()


@pytest.mark.parametrize("mode", ALL_MODES)
@pytest.mark.parametrize("at", [1, 2, 3])
def test_thresholds_off_a_16_byte_boundary(sg, mode, at):
    """A threshold array that starts anywhere in a larger one."""
    import torch
    rng = np.random.default_rng(5)
    batch = workloads.concat([program(total, 7, 9, 0.2, rng) for total in (1, 33, 129, 513)])
    h = sg.sync_load_programs(batch)
    thr = sg.sync_eval_thresholds(h, mode)
    buf = torch.full((thr.numel() + 8,), 1 << 20, dtype=torch.int32, device=thr.device)
    off = buf[at:at + thr.numel()]
    off.copy_(thr)
    assert off.data_ptr() % 16 == 4 * at
    for variant in (oracle.BARRIER, oracle.BARRIER_FREE):
        want = sg.sync_simulate(h, mode, thr, variant=variant)
        got = sg.sync_simulate(h, mode, off, variant=variant)
        for f in ("status", "makespan", "checksum"):
            assert torch.equal(getattr(got, f), getattr(want, f))
        assert not want.status.any()
    h.close()


def device_bytes(sg, h):
    import ctypes
    s = sg.Sizes()
    assert sg.lib().sync_query(h.handle, ctypes.byref(s)) == sg.OK
    return s.device_bytes


@pytest.mark.parametrize("split", [False, True], ids=["whole", "split"])
def test_interval_pool_on_first_use(sg, split, monkeypatch):
    """The iterations' sums are allocated on the first barrier-scheme call
    (unless they are small enough to come with the encoding); a handle that
    may not have them walks, with the same results; one that may takes them
    once."""
    if split:
        monkeypatch.setenv("SYNCGB_SPLIT_MIN", "1")
    rng = np.random.default_rng(23)
    batch = workloads.concat([program(total, 7, 9, 0.2, rng) for total in (1, 33, 129, 513)] +
                             [workloads.generate("depth2", n_programs=3)])
    # per loop around loops that do not run exactly once: starts and sums of the
    # time and every engine's instances
    entries = 0
    for p in range(batch.n_programs):
        l0, l1 = int(batch.prog_loop_ptr[p]), int(batch.prog_loop_ptr[p + 1])
        trips = [batch.trips[batch.trip_ptr[l]:batch.trip_ptr[l + 1]] for l in range(l0, l1)]
        par = batch.loop_parent[l0:l1]
        once = [l > 0 and bool((trips[l] == 1).all()) for l in range(l1 - l0)]
        for l in range(l1 - l0 - 1, 0, -1):
            if not once[l]:
                once[par[l]] = False
        for l in range(l1 - l0):
            if any(par[c] == l and not once[c] for c in range(l + 1, l1 - l0)):
                entries += (1 + int(batch.prog_n_engines[p])) * (2 * int(trips[l].sum()) + 1)
    h = sg.sync_load_programs(batch)
    with_pool = h.sizes.device_bytes
    h.close()
    monkeypatch.setenv("SYNCGB_INTERVAL_POOL", "0")
    h = sg.sync_load_programs(batch)
    assert abs(with_pool - h.sizes.device_bytes - 4 * entries) < 512      # (alignment)
    assert (h.sizes.n_split_programs > 0) == split
    P, prm = batch.n_programs, sg.SimParams()
    thr = sg.sync_eval_thresholds(h, oracle.PERLOOP)
    sg.sync_simulate(h, oracle.PERLOOP, thr)             # barrier-free: the pieces' own scratch
    loaded = device_bytes(sg, h)
    ref = oracle.simulate(batch, oracle.thresholds(batch, oracle.PERLOOP), oracle.PERLOOP, oracle.BARRIER)
    for limit, held in (("0", 0), (str(4 * entries - 1), 0), (str(4 * entries), 4 * entries), (None, 4 * entries),
                        ("0", 4 * entries)):
        if limit is None:
            monkeypatch.delenv("SYNCGB_INTERVAL_POOL")
        else:
            monkeypatch.setenv("SYNCGB_INTERVAL_POOL", limit)
        for r in (sg.sync_simulate(h, oracle.PERLOOP, thr, prm, oracle.BARRIER),
                  sg.sync_simulate_fused(h, oracle.PERLOOP, prm, oracle.BARRIER)):
            assert np.array_equal(r.status.cpu().numpy()[:P], ref.status)
            assert np.array_equal(r.makespan.cpu().numpy()[:P], ref.makespan)
            assert np.array_equal(r.checksum.cpu().numpy()[:P].view(np.uint64), ref.checksum)
        assert device_bytes(sg, h) - loaded == held, limit
    h.close()


@pytest.mark.parametrize("programs", [3, 1217])
@pytest.mark.parametrize("by", ["0", "1", None], ids=["walk", "intervals", "estimate"])
def test_walked_beside_planned(sg, by, programs, monkeypatch):
    """Programs on both sides of the estimate in one batch, few and many
    (more than 8 an SM), and each scheme for all of them."""
    if by is None:
        monkeypatch.delenv("SYNCGB_INTERVALS")
    else:
        monkeypatch.setenv("SYNCGB_INTERVALS", by)
    rng = np.random.default_rng(31)
    some = workloads.concat([program(total, 7, 9, 0.2, rng) for total in (1, 40, 400)])
    batch = workloads.concat([some] * (programs // 3) + [workloads.generate("depth2", n_programs=2)])
    compare_all(sg, batch, modes=[oracle.PERLOOP])
