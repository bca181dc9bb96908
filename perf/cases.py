"""The measured cases: what a program that uses this library has it do.

A case names a batch (a configuration of `workloads`, a number of programs)
and the calls made on it.  The batch and its handle are what a caller keeps;
the calls are one pass:

  step      thresholds, the minimality check, and both simulations -- the
            comparison of the two synchronisation schemes on a batch
  verify    thresholds and check alone (a compiler checking its wait values)
  timeline  thresholds and both simulations with every instance's issue and
            retire time (somebody looks at the schedule)
  engines   the per-engine allocation: its thresholds, its barrier-free
            simulation, and the unrolled program it is compared with
  fused     both simulations with the wait values computed and checked inside
            them, no threshold array
  load      a batch from host arrays: load, thresholds, free (a stream of
            batches, each used once)

Everything computed is an integer, so outputs are compared exactly.
"""
import math
from dataclasses import replace

import numpy as np
import torch

import paper_2608_13757_gb300 as sg
import workloads

MODES = {"count": sg.THR_COUNT, "perloop": sg.THR_PERLOOP, "perengine": sg.THR_PERENGINE}

# Mean pairs, instances and dependencies per program of each configuration
# (measured on its default size), for work() and for the sizes of draw().
PER_PROGRAM = {
    "small": (48, 96, 3),
    "depth2": (8683, 17366, 16),
    "gemm": (143360, 1247232, 33),
    "attention": (1208320, 804864, 23),
    "chain": (5734, 19145, 12.4),
    "syncbound": (2772, 1723, 4.2),
    "trees": (248, 374, 12.3),
}

# Branching loop trees with conditionals, several loops per body and ragged
# trips; one nested dependency in ten lies outside the allocatable cases, so
# programs that hold one take the barrier fallback.
TREES = dict(engines_lo=2, engines_hi=6, max_depth=3, loops_lo=1, loops_hi=6, body_lo=0, body_hi=8, trip_lo=0,
             trip_hi=12, cond_permille=200, lat_lo=1, lat_hi=256, dep_permille=450, max_deps_per_cons=2,
             nest_far_permille=100)


def _case(name, call, config, programs, mode):
    return {"name": name, "call": call, "config": config, "programs": programs, "mode": mode}


def listed():
    return [
        # one small kernel: latency and launches
        _case("small step", "step", "small", 1, "perloop"),
        # one large kernel (a tiled matmul), its schedule looked at
        _case("gemm timeline", "timeline", "gemm", 1, "perloop"),
        # the attention kernels of a model
        _case("attention step", "step", "attention", 256, "perloop"),
        # a sweep over tile shapes: doubly nested loops with redrawn trips
        _case("depth2 step", "step", "depth2", 4096, "perloop"),
        # the same programs, values never stored
        _case("depth2 fused", "fused", "depth2", 1500, "perloop"),
        # an ordinary batch of a compiler's kernels, odd size, paper's base encoding
        _case("chain step 777", "step", "chain", 777, "count"),
        # the largest batch
        _case("chain step 65536", "step", "chain", 65536, "perloop"),
        # wait values only, a large batch of odd size
        _case("chain verify 49999", "verify", "chain", 49999, "perloop"),
        # the per-engine allocation against the unrolled program
        _case("chain engines 4096", "engines", "chain", 4096, "perengine"),
        # batches streamed from the host, each used once
        _case("chain load 8192", "load", "chain", 8192, "perloop"),
        # synchronisation-bound code: conditionals around one instruction
        _case("syncbound step", "step", "syncbound", 65536, "perloop"),
        # a corpus of branching programs, some with the barrier fallback
        _case("trees step", "step", "trees", 6001, "count"),
    ]


# per configuration: smallest and largest number of programs drawn, and the calls
_RANGES = {
    "small": (1, 5000, ("step", "timeline", "engines", "fused")),
    "depth2": (1, 4096, ("step", "verify", "timeline", "engines", "fused", "load")),
    "gemm": (1, 6, ("step", "timeline")),
    "attention": (1, 256, ("step",)),
    "chain": (1, 65536, ("step", "verify", "load")),
    "syncbound": (1, 65536, ("step", "verify")),
    "trees": (1, 12000, ("step", "verify", "timeline", "load")),
}


def draw(rng):
    config = rng.choice(sorted(_RANGES))
    lo, hi, calls = _RANGES[config]
    call = rng.choice(calls)
    if call in ("engines", "fused", "timeline", "load"):
        hi = min(hi, 8192)
    programs = max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))
    mode = "perengine" if call == "engines" else rng.choice(("count", "perloop"))
    c = _case("", call, config, programs, mode)
    del c["name"]
    c["first"] = rng.randrange(1000)          # other programs of the same configuration
    return c


_base = {}          # the last case's batch before a seed's changes


def _batch(case, seed):
    """The case's programs with the seed's latencies and trip counts.  Matmul, attention and small kernels have one
    shape, and the generator draws their latencies.  The others are drawn for the case; the seed turns each loop's
    trip counts by an offset of its own, which keeps the number of instances, and draws the latencies."""
    config, n, first = case["config"], case["programs"], case.get("first", 0)
    if config in ("small", "gemm", "attention"):
        return workloads.generate(config, n, first_program=first, seed=0x5EED0000 + int(seed))
    key = (config, n, first)
    if key not in _base:
        _base.clear()
        if config == "trees":
            _base[key] = workloads.random_trees(0x5EED, n, workloads.tree_params(**TREES), first_program=first)
            _base[key].nonalloc_policy = sg.NONALLOC_BARRIER
        else:
            _base[key] = workloads.generate(config, n, first_program=first)
    b = _base[key]
    rng = np.random.default_rng(int(seed))
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ptr = torch.from_numpy(b.trip_ptr).to(dev)
    size = ptr[1:] - ptr[:-1]
    turn = torch.from_numpy(rng.integers(0, 1 << 30, b.n_loops)).to(dev) % size.clamp(min=1)
    loop = torch.repeat_interleave(torch.arange(b.n_loops, device=dev), size)
    at = torch.arange(len(b.trips), device=dev) - ptr[loop] + turn[loop]
    at = ptr[loop] + torch.where(at >= size[loop], at - size[loop], at)
    trips = torch.from_numpy(b.trips).to(dev)[at].cpu().numpy()
    return replace(b, trips=trips, instr_latency=rng.integers(1, 257, b.n_instrs).astype(np.int32))


def _outputs(h, timeline):
    P = max(h.sizes.n_programs, 1)
    out = sg.SimOutputs(torch.empty(P, dtype=torch.int32, device="cuda"),
                        torch.empty(P, dtype=torch.int64, device="cuda"),
                        torch.empty(P, dtype=torch.int32, device="cuda"))
    if timeline:
        n = max(h.sizes.n_instances, 1)
        out.issue = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        out.retire = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    return out


def prepare(case, seed):
    batch = _batch(case, seed)
    st = {"call": case["call"], "mode": MODES[case["mode"]], "params": sg.SimParams()}
    if case["call"] == "load":
        st["batch"] = batch
        return st
    h = st["h"] = sg.sync_load_programs(batch)
    tl = case["call"] == "timeline"
    if case["call"] != "fused":
        st["thr"] = torch.empty(max(h.sizes.n_pairs_padded, 4), dtype=torch.int32, device="cuda")
    if case["call"] != "verify":
        st["a"], st["b"] = _outputs(h, tl), _outputs(h, tl)
    st["checks"] = [(torch.empty(2, dtype=torch.int64, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda"))
                    for _ in range(2)]
    return st


def _sim(o):
    got = {"makespan": o.makespan, "checksum": o.checksum, "status": o.status}
    if o.issue is not None:
        got["issue"], got["retire"] = o.issue, o.retire
    return got


def run(st):
    call, mode, prm = st["call"], st["mode"], st["params"]
    if call == "load":
        h = sg.sync_load_programs(st["batch"])
        thr = sg.sync_eval_thresholds(h, mode)
        h.close()
        return {"thr": thr}
    h = st["h"]
    got = {}
    if call == "fused":
        (c0, f0), (c1, f1) = st["checks"]
        sg.sync_simulate_fused(h, mode, prm, sg.SIM_BARRIER_FREE, check=True, out=st["a"], counts=c0, first_bad=f0)
        sg.sync_simulate_fused(h, mode, prm, sg.SIM_BARRIER, check=True, out=st["b"], counts=c1, first_bad=f1)
        return {"free": _sim(st["a"]), "barrier": _sim(st["b"]), "counts": [c0, c1], "first_bad": [f0, f1]}
    thr = got["thr"] = sg.sync_eval_thresholds(h, mode, out=st["thr"])
    if call in ("step", "verify"):
        c, f = st["checks"][0]
        got["counts"], got["first_bad"] = sg.sync_check_minimal(h, mode, thr, counts=c, first_bad=f)
    if call == "verify":
        return got
    other = sg.SIM_UNROLLED if call == "engines" else sg.SIM_BARRIER
    got["free"] = _sim(sg.sync_simulate(h, mode, thr, prm, sg.SIM_BARRIER_FREE, out=st["a"]))
    got["unrolled" if call == "engines" else "barrier"] = _sim(sg.sync_simulate(h, mode, thr, prm, other, out=st["b"]))
    return got


def work(case):
    """4 bytes per threshold written, and read by each call that takes them;
    per-program results; 8 bytes per instance and timeline.  The encoding a
    call reads is smaller than these and depends on the batch.  Operations:
    12 integer ones per instance and simulation, 2 per pair and simulation,
    4 per pair for a threshold and for its check."""
    pairs, inst, deps = (x * case["programs"] for x in PER_PROGRAM[case["config"]])
    call = case["call"]
    sims = {"step": 2, "timeline": 2, "engines": 2, "fused": 2}.get(call, 0)
    evals = {"step": 2, "verify": 2, "fused": 4}.get(call, 1)
    touched = 0 if call == "fused" else 1 + (call in ("step", "verify")) + sims
    byt = 4.0 * pairs * touched + 16.0 * case["programs"] * sims + 80.0 * deps
    if call == "timeline":
        byt += 8.0 * inst * sims
    if call == "load":
        byt += 4.0 * inst / 16                 # the trip counts, about one per 16 instances
    return {"bytes": byt, "flops": sims * (12.0 * inst + 2.0 * pairs) + 4.0 * pairs * evals}


def tolerance(case):
    return "exact"


# ------------------------------------------------------- results in 64 bits

_MAX_DEPS, _MAX_PAIRS, _MAX_INST = 12000, 6_000_000, 250_000


class _Program:
    """One program of a batch: its loops' trip prefix sums and bodies."""

    def __init__(self, b, p):
        l0, l1 = int(b.prog_loop_ptr[p]), int(b.prog_loop_ptr[p + 1])
        x0, x1 = int(b.prog_instr_ptr[p]), int(b.prog_instr_ptr[p + 1])
        d0, d1 = int(b.prog_dep_ptr[p]), int(b.prog_dep_ptr[p + 1])
        self.ne = int(b.prog_n_engines[p])
        self.par = b.loop_parent[l0:l1].tolist()
        self.lpos = b.loop_pos[l0:l1].tolist()
        self.rp = [np.concatenate([[0], np.cumsum(b.trips[b.trip_ptr[l]:b.trip_ptr[l + 1]], dtype=np.int64)])
                   for l in range(l0, l1)]
        self.total = [int(r[-1]) for r in self.rp]
        self.il, self.ip = b.instr_loop[x0:x1].tolist(), b.instr_pos[x0:x1].tolist()
        self.ie, self.lat = b.instr_engine[x0:x1].tolist(), b.instr_latency[x0:x1].tolist()
        self.deps = list(zip(b.dep_prod[d0:d1].tolist(), b.dep_cons[d0:d1].tolist(), b.dep_k[d0:d1].tolist()))
        self.depth = [0] * (l1 - l0)
        for l in range(1, l1 - l0):
            self.depth[l] = self.depth[self.par[l]] + 1
        self.body = [[] for _ in range(l1 - l0)]
        for x, l in enumerate(self.il):
            self.body[l].append((self.ip[x], x, True))
        for l in range(1, l1 - l0):
            self.body[self.par[l]].append((self.lpos[l], l, False))
        for body in self.body:
            body.sort()

    def dep(self, d):
        """(the common loop, its children towards producer and consumer, whether a barrier stands for it)"""
        px, cx, k = d
        a, c, up, down = self.il[px], self.il[cx], -1, -1
        while self.depth[a] > self.depth[c]:
            down, a = a, self.par[a]
        while self.depth[c] > self.depth[a]:
            up, c = c, self.par[c]
        while a != c:
            down, a, up, c = a, self.par[a], c, self.par[c]
        if down < 0:
            return a, down, up, False
        forward = (self.ip[cx] if up < 0 else self.lpos[up]) > self.lpos[down]
        return a, down, up, k != (0 if forward else 1)

    def producers(self, d):
        """Per consumer instance, the producer instances that Eq. (1) requires: those in iterations of the common
        loop up to the consumer's less the offset, in the same trip; none if there is no such iteration."""
        px, cx, k = d
        s, _, _, barrier = self.dep(d)
        g = np.arange(self.total[self.il[cx]], dtype=np.int64)
        if barrier:
            return np.zeros_like(g)
        l = self.il[cx]
        while l != s:
            g = np.searchsorted(self.rp[l], g, side="right") - 1
            l = self.par[l]
        start = self.rp[s][np.searchsorted(self.rp[s], g, side="right") - 1]
        x, chain, l = g - k + 1, [], self.il[px]
        while l != s:
            chain.append(l)
            l = self.par[l]
        hit = x > start
        x = np.where(hit, x, 0)
        for l in reversed(chain):
            x = self.rp[l][x]
        return np.where(hit, x, 0)


def _encoded(pr, d, c, mode):
    """Eq. (5) of the paper for the per-(loop, engine) semaphore, else the count."""
    if mode != sg.THR_PERLOOP:
        return c
    px = d[0]
    same = sorted(pr.ip[x] for x in range(len(pr.il)) if pr.il[x] == pr.il[px] and pr.ie[x] == pr.ie[px])
    n, k = len(same), same.index(pr.ip[px]) + 1
    return np.where(c > 0, n * c - (n - k), 0)


def _simulated(pr, want, cw, barrier, timeline):
    """The timing model, instance by instance in program order: (makespan, checksum, issue, retire), or None where a
    wait names an instance later in that order."""
    t, last, count = [0] * pr.ne, [0] * pr.ne, [0] * pr.ne
    times = [[] for _ in pr.il]
    terms = []
    waits = [[] for _ in pr.il]
    ends = set()
    for i, d in enumerate(pr.deps):
        s, _, _, bar = pr.dep(d)
        if bar:
            ends.add(s)
        else:
            waits[d[1]].append((d[0], want[i].tolist()))
    start = 1 if barrier else 3

    def all_engines():
        r = max(max(a, b) for a, b in zip(t, last)) + 32
        t[:] = [r] * pr.ne

    def walk(l, g):
        for _, i, instr in pr.body[l]:
            if instr:
                e = pr.ie[i]
                at = t[e] + (0 if barrier else cw * len(waits[i]))
                for px, c in waits[i]:
                    if c[g] > len(times[px]):
                        return False
                    if c[g]:
                        at = max(at, times[px][c[g] - 1][1])
                done = max(at + pr.lat[i], last[e])
                t[e], last[e] = at + 1, done
                count[e] += 1
                times[i].append((at, done))
                terms.append((at, done, e, count[e]))
                continue
            if barrier:
                all_engines()
            else:
                t[:] = [v + 1 for v in t]
            for j in range(int(pr.rp[i][g]), int(pr.rp[i][g + 1])):
                t[:] = [v + start for v in t]
                if not walk(i, j):
                    return False
                if barrier or i in ends:
                    all_engines()
        return True

    if not walk(0, 0):
        return None
    a = np.array(terms, dtype=np.int64).reshape(-1, 4)
    m = np.int64(0xFFFFFFFF)
    u = ((a[:, 0] ^ ((a[:, 3] * 0x9E3779B9 + a[:, 2]) & m)) * 0x85EBCA6B) & m
    v = ((a[:, 1] ^ ((a[:, 3] * 0xC2B2AE35 + a[:, 2]) & m)) * 0x27D4EB2F) & m
    u, v = u ^ (u >> 13), v ^ (v >> 15)
    mix = (u.astype(np.uint64) << np.uint64(32)) | v.astype(np.uint64)
    flat = np.array([x for xs in times for x in xs], dtype=np.int64).reshape(-1, 2) if timeline else None
    return max(max(p, q) for p, q in zip(t, last)), mix.sum(dtype=np.uint64), flat


def exact(case, seed):
    if case["call"] == "engines":
        return None
    pairs, inst, deps = (x * case["programs"] for x in PER_PROGRAM[case["config"]])
    if deps > _MAX_DEPS or pairs > _MAX_PAIRS:
        return None
    b, mode, call = _batch(case, seed), MODES[case["mode"]], case["call"]
    programs = [_Program(b, p) for p in range(b.n_programs)]
    want = [[pr.producers(d) for d in pr.deps] for pr in programs]
    parts = []
    for pr, cs in zip(programs, want):
        for d, c in zip(pr.deps, cs):
            parts += [_encoded(pr, d, c, mode), np.zeros(-len(c) % 4, dtype=np.int64)]
    thr = np.concatenate(parts) if parts else np.zeros(0, dtype=np.int64)
    thr = np.concatenate([thr, np.zeros(max(0, 4 - len(thr)), dtype=np.int64)]).astype(np.int32)
    none = np.zeros(2, dtype=np.int64), np.full(1, -1, dtype=np.int64)
    if call == "load":
        return {"thr": thr}
    got = {} if call == "fused" else {"thr": thr}
    if call == "verify" or call == "step":
        got["counts"], got["first_bad"] = none
    if call == "fused":
        got["counts"], got["first_bad"] = [none[0]] * 2, [none[1]] * 2
    if call == "verify":
        return got
    for name, barrier in (("free", False), ("barrier", True)):
        got[name] = None
        if inst > _MAX_INST:
            continue
        sims = [_simulated(pr, cs, 3 if mode == sg.THR_COUNT else 5, barrier, call == "timeline")
                for pr, cs in zip(programs, want)]
        if any(s is None for s in sims):
            continue
        got[name] = {"makespan": np.array([s[0] for s in sims], dtype=np.int32),
                     "checksum": np.array([s[1] for s in sims], dtype=np.uint64).view(np.int64),
                     "status": np.zeros(len(sims), dtype=np.int32)}
        if call == "timeline":
            flat = np.concatenate([s[2] for s in sims]).astype(np.int32)
            got[name]["issue"], got[name]["retire"] = np.ascontiguousarray(flat[:, 0]), np.ascontiguousarray(flat[:, 1])
    return got
