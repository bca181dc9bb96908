// Barrier scheme by intervals.
//
// The barriers (before every loop statement, at the end of every iteration)
// cut a program's run into intervals.  An interval starts at a release: every
// engine at the same time, everything earlier retired.  So a wait on an
// increment published before the interval never binds, and when each of a
// segment's waits either is such a wait on every visit or names its own
// producer's increment of the same visit on every visit, the segment has one
// schedule relative to its start.  Start times are then sums of per-loop
// constants: with K_l the duration of an iteration of loop l without its
// moving child loops (those that do not run exactly once on every visit), its
// first x iterations take
//     P_l(x) = K_l * x + sum over its moving children c of P_c(R_c(x)),
// R_c the trip prefix sums.  Positions in the engines' streams are the same
// sums over instance counts.  Three stages:
//   plan     (a warp per program) the waits classified on their first visit,
//            every segment's schedule by in-order issue of its engines, P
//            from the inside out and the iterations' starts from the outside
//            in, for the loops with moving children;
//   tile     (a warp per tile of a loop's iterations) every wait compared
//            with its class, every instance's times and checksum term;
//   a program with a wait outside its class, or whose segment cannot be
//   scheduled, is swept instead (k_sweep), which gives its verdict.
// A program whose walk takes less than its plan is walked too (enc.h has the
// rule).  Nothing is serial but a program's plan.  What bounds a tile is its
// integer instructions -- 14 per instance and lane for the times and the
// checksum, 7 per wait -- and the latency of its prologue.  Barrier simulation,
// walked / by intervals: 65536 chain programs (1.25e9 instances) 15.1 / 4.7 ms
// (plans 0.6, waits 1.6, times 2.2), 65536 sync-bound ones 35.2 / 3.6, 256
// attention programs 14.3 / 0.87, 4096 depth-2 ones 4.1 / 0.36, the GEMM 2.7 /
// 0.18.  These are repeated calls: the first one on a handle also lays out the
// positions in the engines' streams, which depend on the batch alone (chain
// 5.1 ms, pool allocation included; 3000 branching trees 0.62 instead of 0.35,
// cold caches included).  On every call they would take 0.34 ms of the chain's.
#pragma once

#include "cost.cuh"
#include "waitval.cuh"

namespace syncgb {
namespace {

constexpr unsigned kBarFull = 0xffffffffu;
constexpr int kBarU = 4;                    // iterations per lane at a time
// The interval sweep: resident CTAs per SM, and the shared memory of a CTA's
// semaphore rings (its walk is for the programs left over).  65536 chain
// programs: 5.2 ms at 3 CTAs (80 registers), 4.8 at 4, 4.7 at 5, 4.8 at 6;
// 777 of them 0.22, 0.24, 0.29, 0.33.
constexpr int kBarCtas = 4;

__device__ __forceinline__ unsigned long long inst_mix(uint32_t issue, uint32_t retire, uint32_t a1, uint32_t a2) {
  uint32_t x = (issue ^ a1) * 0x85EBCA6Bu;
  x ^= x >> 13;
  uint32_t y = (retire ^ a2) * 0x27D4EB2Fu;
  y ^= y >> 15;
  return ((unsigned long long)x << 32) | y;
}
constexpr uint32_t kMixA = 0x9E3779B9u, kMixB = 0xC2B2AE35u;

struct BarProg { int32_t le_base, loop_base, ne; };
__device__ __forceinline__ BarProg bar_prog(const ProgInfo& pi) { return BarProg{pi.le_base, pi.loop_base, pi.ne}; }

__device__ __forceinline__ int32_t bar_row(const BarProg& b, int l) { return b.le_base + (l - b.loop_base) * b.ne; }

// Quantity q (0 = time, 1 + e = instances of engine e) of one iteration of
// loop l, and before it in its parent's (moving loops excluded).  ko and F
// are written by other warps of the launch: read past L1.
__device__ __forceinline__ uint32_t bar_k(const SweepArgs& a, const BarProg& b, int l, int q) {
  return q == 0 ? (uint32_t)__ldcg(a.bar.ko + l).x : (uint32_t)__ldg(a.bar.rowc + bar_row(b, l) + q - 1).y;
}
__device__ __forceinline__ uint32_t bar_off(const SweepArgs& a, const BarProg& b, int l, int q) {
  return q == 0 ? (uint32_t)__ldcg(a.bar.ko + l).y : (uint32_t)__ldg(a.bar.rowc + bar_row(b, l) + q - 1).x;
}
__device__ __forceinline__ int64_t bar_rp(const int4 ax) {
  return (int64_t)(((uint64_t)(uint32_t)ax.y << 32) | (uint32_t)ax.x);
}

// Arrays of a loop with moving children: starts and sums of quantity q.
__device__ __forceinline__ int32_t* bar_starts(const SweepArgs& a, int64_t foff, int32_t total, int q) {
  return a.bar.F + foff + (int64_t)q * total;
}
__device__ __forceinline__ int32_t* bar_sums(const SweepArgs& a, const BarProg& b, int64_t foff, int32_t total, int q) {
  return a.bar.F + foff + (int64_t)(1 + b.ne) * total + (int64_t)q * (total + 1);
}

// P_l(x1) - P_l(x0).
__device__ __forceinline__ uint32_t bar_span(const SweepArgs& a, const BarProg& b, int l, int32_t x0, int32_t x1, int q) {
  const int64_t foff = a.bar.bl[l].foff;
  if (foff < 0) return bar_k(a, b, l, q) * (uint32_t)(x1 - x0);
  const int32_t* P = bar_sums(a, b, foff, a.loop[l].total, q);
  return (uint32_t)__ldcg(P + x1) - (uint32_t)__ldcg(P + x0);
}

// What the moving children (`all`: every child) of a loop at plan items
// [i0, i1) add in its iteration j.
__device__ __noinline__ uint32_t bar_children(const SweepArgs& a, const BarProg& b, int i0, int i1, int32_t j, int q,
                                              bool all) {
  uint32_t acc = 0;
  for (int i = i0; i < i1; ++i) {
    const int4 v = __ldg(a.plan + i);
    if (v.x != ITEM_LOOP || (!all && a.bar.bl[v.y].host != v.y)) continue;
    const int64_t rp = bar_rp(__ldg(a.paux + i));
    acc += bar_span(a, b, v.y, __ldg(a.rowptr + rp + j), __ldg(a.rowptr + rp + j + 1), q);
  }
  return acc;
}

// Quantity q at the start of iteration g (lo: the first of its trip, j: its
// parent's iteration) of loop l, its own host and not the top level.
__device__ __forceinline__ uint32_t bar_start(const SweepArgs& a, const BarProg& b, int l, const LoopInfo& L,
                                              const BarLoop& B, int32_t j, int32_t lo, int32_t g, int q) {
  uint32_t v = bar_off(a, b, l, q) + (uint32_t)__ldcg(bar_starts(a, a.bar.bl[L.parent].foff, L.n_parent, q) + j);
  if (B.esib > 0) v += bar_children(a, b, __ldg(a.plan_ptr + L.parent), B.item, j, q, false);
  return v + bar_span(a, b, l, lo, g, q);
}

// The row (parent iteration) of iteration g in the trip prefix sums rp[0..n]:
// the largest j < n with rp[j] <= g.
__device__ __forceinline__ int32_t bar_row_of(const int32_t* __restrict__ rp, int32_t n, int32_t g) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo + 1) >> 1);
    if (__ldg(rp + mid) <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}
// The same by the whole warp for one g (32 probes a step).
__device__ __forceinline__ int32_t bar_row_warp(const int32_t* __restrict__ rp, int32_t n, int32_t g, int lane) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t step = (hi - lo + 31) / 32;
    const int64_t at = lo + (int64_t)(lane + 1) * step;
    const bool le = at <= hi && __ldg(rp + at) <= g;
    const int c = __popc(__ballot_sync(kBarFull, le));
    const int32_t nlo = lo + c * step;
    hi = min(hi, nlo + step - 1);
    lo = nlo;
  }
  return lo;
}
// Rows j and their first iterations lo of 32 consecutive iterations from
// `first` (the lanes' g, clamped to the last one), from row j0 at or before
// the first lane's.  Usually no row that starts among them is empty: each
// start then sets its own bit, and a lane counts the bits up to it.
__device__ __forceinline__ void bar_rows(const int32_t* __restrict__ rp, int32_t n, int32_t first, int32_t g, int32_t j0,
                                         int lane, int32_t& j, int32_t& lo) {
  const bool row = j0 + 1 + lane < n;
  int32_t v = row ? __ldg(rp + j0 + 1 + lane) : 0x7fffffff;
  const int32_t at = v - first;
  const bool in = row && at >= 0 && at < 32;
  const unsigned starts = __reduce_or_sync(kBarFull, in ? 1u << at : 0u);
  const unsigned who = __ballot_sync(kBarFull, in);
  const unsigned past = __ballot_sync(kBarFull, !row || at >= 32);
  const unsigned skip = ~(who | past);      // rows that start before the first iteration: the last of them holds it
  if (past != 0 && __popc(starts) == __popc(who)) {
    const unsigned le = starts & (2u * (1u << (g - first)) - 1u);
    const int32_t jf = j0 + __popc(skip);
    j = jf + __popc(le);
    lo = le ? first + 31 - __clz(le) : __ldg(rp + jf);
    return;
  }
  j = -1;
  for (int32_t base = j0;; v = base + 1 + lane < n ? __ldg(rp + base + 1 + lane) : 0x7fffffff) {
    int c = 0;                              // row starts <= g among the next 32 rows'
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
      if (__shfl_sync(kBarFull, v, c + s - 1) <= g) c += s;
    if (__shfl_sync(kBarFull, v, c) <= g) ++c;
    if (j < 0 && c < 32) j = base + c;
    if (!__ballot_sync(kBarFull, j < 0)) break;
    base += 32;
  }
  lo = __ldg(rp + j);
}

// The sums of loop l, quantities [q0, q1), by one warp; its children's are
// there.
__device__ void bar_fill_sums(const SweepArgs& a, const BarProg& b, int l, int q0, int q1, int lane) {
  const BarLoop B = a.bar.bl[l];
  const int32_t total = a.loop[l].total;
  const int i0 = __ldg(a.plan_ptr + l), i1 = __ldg(a.plan_ptr + l + 1);
  for (int32_t gb = 0; gb <= total; gb += 128)
    for (int q = q0; q < q1; ++q) {
      uint32_t v[4];
      const uint32_t K = bar_k(a, b, l, q);
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = K * (uint32_t)min(gb + 32 * u + lane, total);
      for (int i = i0; i < i1; ++i) {
        const int4 it = __ldg(a.plan + i);
        if (it.x != ITEM_LOOP || a.bar.bl[it.y].host != it.y) continue;
        const int32_t* rp = a.rowptr + bar_rp(__ldg(a.paux + i));
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] += bar_span(a, b, it.y, 0, __ldg(rp + min(gb + 32 * u + lane, total)), q);
      }
      int32_t* P = bar_sums(a, b, B.foff, total, q);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (gb + 32 * u + lane <= total) __stcg(P + gb + 32 * u + lane, (int32_t)v[u]);
    }
  __syncwarp();
}

// The starts of loop l (not the top level), quantities [q0, q1), by one
// warp; its sums and its parent's starts are there.
__device__ void bar_fill_starts(const SweepArgs& a, const BarProg& b, int l, int q0, int q1, int lane) {
  const LoopInfo L = a.loop[l];
  const BarLoop B = a.bar.bl[l];
  const int32_t* rp = a.rowptr + L.rowptr_off;
  int32_t j0 = 0;
  for (int32_t gb = 0; gb < L.total; gb += 32) {
    const int32_t g = min(gb + lane, L.total - 1);
    int32_t j, lo;
    bar_rows(rp, L.n_parent, gb, g, j0, lane, j, lo);
    j0 = __shfl_sync(kBarFull, j, 31);
    for (int q = q0; q < q1; ++q) {
      const uint32_t v = bar_start(a, b, l, L, B, j, lo, g, q);
      if (gb + lane < L.total) __stcg(bar_starts(a, B.foff, L.total, q) + g, (int32_t)v);
    }
  }
  __syncwarp();
}

// Both for every loop of a program that has them.
__device__ void bar_fill(const SweepArgs& a, const ProgInfo& pi, int q0, int q1, int lane) {
  const BarProg b = bar_prog(pi);
  for (int l = pi.loop_base + pi.nloops - 1; l >= pi.loop_base; --l)
    if (a.bar.bl[l].foff >= 0 && a.loop[l].total > 0) bar_fill_sums(a, b, l, q0, q1, lane);
  const int64_t top = a.bar.bl[pi.loop_base].foff;
  if (top >= 0 && lane == 0)
    for (int q = q0; q < q1; ++q) __stcg(bar_starts(a, top, 1, q), 0);
  __syncwarp();
  for (int l = pi.loop_base + 1; l < pi.loop_base + pi.nloops; ++l)
    if (a.bar.bl[l].foff >= 0 && a.loop[l].total > 0) bar_fill_starts(a, b, l, q0, q1, lane);
}

// Instances of engine e before loop l's iteration g, by one thread.
__device__ __noinline__ uint32_t bar_count_at(const SweepArgs& a, const BarProg& b, int l, int32_t g, int e) {
  const int h = a.bar.bl[l].host;
  uint32_t v = 0;
  if (l != h) {                             // in an iteration of its host
    int c = l;
    while (a.loop[c].parent != h) c = a.loop[c].parent;
    v = (uint32_t)__ldg(a.bar.rowc + bar_row(b, l) + e).x;
    if (a.bar.bl[c].esib > 0) v += bar_children(a, b, __ldg(a.plan_ptr + h), a.bar.bl[c].item, g, 1 + e, false);
  }
  const LoopInfo H = a.loop[h];
  const BarLoop B = a.bar.bl[h];
  if (H.parent < 0) return v;
  if (B.foff >= 0) return v + (uint32_t)__ldcg(bar_starts(a, B.foff, H.total, 1 + e) + g);
  const int32_t* rp = a.rowptr + H.rowptr_off;
  const int32_t j = bar_row_of(rp, H.n_parent, g);
  return v + bar_start(a, b, h, H, B, j, __ldg(rp + j), g, 1 + e);
}

// The producer engine's instances before the consumer's iteration g and its
// child loops so far (per-engine waits).
__device__ __forceinline__ int32_t bar_engine_pub(const SweepArgs& a, const BarProg& b, const BarDep& bd, int32_t g) {
  uint32_t v = bar_count_at(a, b, bd.cons_loop, g, bd.ep);
  if (bd.cons_item >= 0)
    v += bar_children(a, b, __ldg(a.plan_ptr + bd.cons_loop), bd.cons_item + 1, g, 1 + bd.ep, true);
  return (int32_t)v;
}

// Increments of dependency r's semaphore published at the start of the
// consumer's interval (its S-iteration gs), and its own producer's increment
// of the same iteration.  pe (per-engine semaphores): the producer engine's
// instances before the consumer's iteration and its child loops so far.
template <int MODE>
__device__ __forceinline__ void bar_pub(const SweepArgs& a, const DepInfo& D, const BarDep& bd, int32_t gs, int32_t pe,
                                        int32_t& pub, int32_t& own) {
  if (MODE == SYNC_THR_PERENGINE) {
    pub = pe + bd.b2;
    own = pe + D.K;
    return;
  }
  const int32_t X = bd.prod_fixed ? gs + bd.delta : count_down(a.bar, D, gs + bd.delta, a.rowptr);
  if (MODE == SYNC_THR_PERLOOP) {
    pub = D.N * X + bd.b[1];
    own = D.N * gs + D.K;
  } else {
    pub = X + bd.b[0];
    own = gs + 1;
  }
}

// The counts of program p's starts and sums (q >= 1), once per handle.
__device__ __forceinline__ void bar_counts(const SweepArgs& a, int p, const ProgInfo& pi, int lane) {
  if (a.bar.counted[p]) return;
  bar_fill(a, pi, 1, 1 + pi.ne, lane);
  if (lane == 0) a.bar.counted[p] = 1;
}

// The wait value of dependency D at the consumer's iteration g, whose
// S-iteration is gs, computed (fused), and whether Eq. (1)'s minimum is it.
template <int MODE>
__device__ __forceinline__ int32_t bar_value(const SweepArgs& a, const DepInfo& D, int32_t g, int32_t gs, bool& bad) {
  const int32_t st = D.src < 0 ? 0 : __ldg(a.bar.derived + (D.up == 0 ? D.src + g : D.tstart + gs));
  const int32_t T = wait_value(a, D, gs, st, MODE);
  bad = bad || (a.chk_counts && minimum(a, D, gs, st, MODE) != T);
  return T;
}

// The classes of program p's waits, from each one's first visit.  False: a
// wait is neither on an earlier interval nor on its own producer (or, fused,
// differs from the checked minimum: the walk tallies it).
template <int MODE, bool FUSED>
__device__ bool bar_classes(const SweepArgs& a, const ProgInfo& pi, int lane) {
  const BarProg b = bar_prog(pi);
  bool bad = false;
  for (int r = pi.dep0 + lane; r < pi.dep0 + pi.ndep; r += 32) {
    const DepInfo D = a.bar.dep[__ldg(a.bar.ddep + r)];
    if (D.total == 0) { a.bar.bind[r] = 0; continue; }
    const BarDep bd = a.bar.bdep[r];
    const int32_t gs = D.up == 0 || D.src < 0 ? 0 : __ldg(a.bar.derived + D.src);
    const int32_t pe = MODE == SYNC_THR_PERENGINE ? bar_engine_pub(a, b, bd, 0) : 0;
    int32_t pub, own;
    bar_pub<MODE>(a, D, bd, gs, pe, pub, own);
    const int32_t T = FUSED ? bar_value<MODE>(a, D, 0, gs, bad) : __ldg(a.thr + D.seg_off);
    const bool in = T > pub;
    bad = bad || (in && (!bd.in_seg || T != own));
    a.bar.bind[r] = in ? 1 : 0;
  }
  return !__ballot_sync(kBarFull, bad);
}

// The schedules of loop l's segments: every engine in its own lane, in
// rounds (a record issues once its producers in the segment have); at:
// 32 ints of shared memory.  Writes rel of its records, ko.x of l and ko.y
// of its children, whose fixed ones are scheduled.  False: no engine can go
// on.
__device__ bool bar_schedule(const SweepArgs& a, const BarProg& b, int l, volatile int32_t* at, int lane) {
  const bool top = l == b.loop_base;
  const int32_t row = bar_row(b, l);
  int32_t i = lane < b.ne ? __ldg(a.bar.op_ptr + row + lane) : 0;
  int4 rec = lane < b.ne ? __ldg(a.bar.ops + i) : make_int4(OP_END, 0, 0, 0);
  int32_t cst = top ? 0 : a.prm.c_branch;
  int item = __ldg(a.plan_ptr + l);
  for (;;) {
    int32_t t = 0, lr = 0;
    at[lane] = i;
    __syncwarp();
    bool more = rec.x >= 0;
    while (__ballot_sync(kBarFull, more)) {
      bool ready = more;
      int32_t r = 0;
      if (more) {
        for (int j = 0; j < rec.z; ++j) {
          if (!a.bar.bind[rec.w + j]) continue;
          const BarDep bd = a.bar.bdep[rec.w + j];
          if (at[bd.ep] > bd.prod_op) r = max(r, __ldcg(a.bar.rel + bd.prod_op).y - cst);
          else ready = false;
        }
      }
      if (!__ballot_sync(kBarFull, ready)) return false;
      if (ready) {
        const int32_t issue = max(t, r);
        lr = max(issue + rec.y, lr);
        t = issue + a.prm.ii;
        __stcg(a.bar.rel + i, make_int2(cst + issue, cst + lr));
        ++i;
        rec = __ldg(a.bar.ops + i);
        more = rec.x >= 0;
      }
      __syncwarp();
      at[lane] = i;
      __syncwarp();
    }
    const int32_t end = cst + (int32_t)__reduce_max_sync(kBarFull, (unsigned)max(t, lr));
    if (__shfl_sync(kBarFull, rec.x, 0) == OP_END) {
      if (lane == 0) a.bar.ko[l].x = end + (top ? 0 : a.prm.c_barrier);
      break;
    }
    cst = end + a.prm.c_barrier;
    while (__ldg(a.plan + item).x != ITEM_LOOP) ++item;
    const int c = __ldg(a.plan + item++).y;
    if (lane == 0) a.bar.ko[c].y = cst;
    if (a.bar.bl[c].host != c) cst += __ldcg(a.bar.ko + c).x;
    if (lane < b.ne) {
      ++i;
      rec = __ldg(a.bar.ops + i);
    }
  }
  __syncwarp();
  return true;
}

// The schedules of loop h and of the fixed loops in its iterations, inner
// ones first.
__device__ bool bar_schedules(const SweepArgs& a, const ProgInfo& pi, int h, volatile int32_t* at, int lane) {
  const BarProg b = bar_prog(pi);
  bool ok = true;
  for (int l = pi.loop_base + pi.nloops - 1; ok && l >= h; --l)
    if (a.bar.bl[l].host == h) ok = bar_schedule(a, b, l, at, lane);
  return ok;
}

// From the schedules: sums and starts, makespan, the outputs the tiles add to.
__device__ void bar_compose(const SweepArgs& a, int p, const ProgInfo& pi, int lane) {
  const BarProg b = bar_prog(pi);
  bar_fill(a, pi, 0, 1, lane);
  if (lane == 0) {
    a.makespan[p] = (int32_t)bar_span(a, b, pi.loop_base, 0, 1, 0);
    a.status[p] = SYNC_PROG_OK;
    a.checksum[p] = 0;
    a.bar.left[p] = a.bar.bl[pi.loop_base + pi.nloops].tile0 - a.bar.bl[pi.loop_base].tile0;
  }
}

template <int MODE>
__device__ __forceinline__ bool bar_in_time(const SweepArgs& a, const ProgInfo& pi) {
  return time_bound<MODE, true>(pi, a.prm, 0) <= 2147483647ull;
}

// Program p's plan by one warp; false: it has to be swept.
template <int MODE, bool FUSED>
__device__ __noinline__ bool bar_plan(const SweepArgs& a, int p, int32_t* at, int lane) {
  const ProgInfo pi = a.prog[p];
  const BarProg b = bar_prog(pi);
  bool ok = (pi.intervals & a.bar.which) && bar_in_time<MODE>(a, pi);
  if (ok) {
    bar_counts(a, p, pi, lane);
    ok = bar_classes<MODE, FUSED>(a, pi, lane);
  }
  __syncwarp();
  for (int l = pi.loop_base + pi.nloops - 1; ok && l >= pi.loop_base; --l)
    if (a.loop[l].total > 0) ok = bar_schedule(a, b, l, at, lane);
  __syncwarp();
  if (ok) bar_compose(a, p, pi, lane);
  else if (lane == 0) a.bar.left[p] = -1;
  return ok;
}

// One tile by one warp: iterations g0.. of loop l.  Two passes over the
// body's op records (32 at a time, one per lane): the waits, four
// consecutive iterations per lane so that thresholds and S-iterations come
// in 16-byte loads, and the instances, a lane per iteration and kBarU
// iterations per lane, which one broadcast of a record serves.  `at`: 32
// ints of shared memory.  Returns whether a wait is outside its class
// (warp-uniform).
template <int MODE, bool FUSED>
__device__ __forceinline__ bool bar_waits(const SweepArgs& a, const BarProg& b, int32_t g0, int32_t g1,
                                          const int4 op, int32_t* at, int lane) {
  // the chunk's dependencies, one per lane
  const int z = op.x >= 0 ? op.z : 0;
  int pre = z;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kBarFull, pre, o);
    if (lane >= o) pre += v;
  }
  const int total = __shfl_sync(kBarFull, pre, 31);
  pre -= z;
  bool bad = false;
  for (int k0 = 0; k0 < total; k0 += 32) {
    for (int j = max(0, k0 - pre); j < z && pre + j - k0 < 32; ++j) at[pre + j - k0] = op.w + j;
    __syncwarp();
    const int n = min(32, total - k0);
    // limit of the wait value at iteration g: mul * X + add, X = g (kind 0),
    // the S-iteration (1), 0 (2), or counted below S (3)
    int64_t seg = 0, src = 0;
    int32_t mul = 0, add = 0, kind = 0, r = 0;
    if (lane < n) {
      r = at[lane];
      const DepInfo D = a.bar.dep[__ldg(a.bar.ddep + r)];
      const BarDep bd = a.bar.bdep[r];
      const bool in = __ldcg(a.bar.bind + r) != 0;
      seg = D.seg_off;
      src = D.src;
      mul = MODE == SYNC_THR_PERLOOP ? D.N : 1;
      add = in ? (MODE == SYNC_THR_PERLOOP ? D.K : 1) : MODE == SYNC_THR_PERLOOP ? bd.b[1] : bd.b[0];
      if (bd.prod_fixed) add += in ? 0 : mul * bd.delta;
      for (int32_t g = g0; !FUSED && g < g1; g += 32)   // the thresholds' lines, while the others' records load
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.thr + seg + g));
      kind = (!(bd.prod_fixed) ? 3 : bd.cons_fixed ? 0 : D.src < 0 ? 2 : 1) | (in ? 4 : 0);
    }
    __syncwarp();
    for (int k = 0; k < n; ++k) {
      const int kk = __shfl_sync(kBarFull, kind, k);
      const int64_t so = __shfl_sync(kBarFull, seg, k);
      // (thresholds that start off a 16-byte boundary are read one by one)
      if (FUSED || MODE == SYNC_THR_PERENGINE || (kk & 3) == 3 || (reinterpret_cast<uintptr_t>(a.thr) & 15)) {
        const int rr = __shfl_sync(kBarFull, r, k);
        const DepInfo D = a.bar.dep[__ldg(a.bar.ddep + rr)];
        const BarDep bd = a.bar.bdep[rr];
        for (int32_t g = g0 + lane; g < g1; g += 32) {
          const int32_t gs = D.up == 0 ? g : D.src < 0 ? 0 : __ldg(a.bar.derived + D.src + g);
          const int32_t pe = MODE == SYNC_THR_PERENGINE ? bar_engine_pub(a, b, bd, g) : 0;
          int32_t pub, own;
          bar_pub<MODE>(a, D, bd, gs, pe, pub, own);
          const int32_t T = FUSED ? bar_value<MODE>(a, D, g, gs, bad) : __ldg(a.thr + so + g);
          bad = bad || (kk & 4 ? T != own : T > pub);
        }
        continue;
      }
      const int64_t ds = __shfl_sync(kBarFull, src, k);
      const int32_t m = __shfl_sync(kBarFull, mul, k), c = __shfl_sync(kBarFull, add, k);
      // segments and derived arrays start at multiples of 4 entries and are
      // padded to them, and so does a tile
      for (int32_t g = g0 + 4 * lane; g < g1; g += 128) {
        const int4 T = __ldcs(reinterpret_cast<const int4*>(a.thr + so + g));
        int4 X = make_int4(g, g + 1, g + 2, g + 3);
        if ((kk & 3) == 1) X = __ldg(reinterpret_cast<const int4*>(a.bar.derived + ds + g));
        if ((kk & 3) == 2) X = make_int4(0, 0, 0, 0);
        const int32_t d0 = T.x - (m * X.x + c), d1 = T.y - (m * X.y + c), d2 = T.z - (m * X.z + c),
                      d3 = T.w - (m * X.w + c);
        if (kk & 4)
          bad = bad || d0 != 0 || (g + 1 < g1 && d1 != 0) || (g + 2 < g1 && d2 != 0) || (g + 3 < g1 && d3 != 0);
        else
          bad = bad || d0 > 0 || (g + 1 < g1 && d1 > 0) || (g + 2 < g1 && d2 > 0) || (g + 3 < g1 && d3 > 0);
      }
    }
  }
  return bad;
}

// A body's op records 32 at a time, engine by engine: begin(e) before an
// engine's first record or child loop, record(rel.x, rel.y, instance
// offset), child(loop, its rowptr offset).
template <bool TL, class Begin, class Record, class Child>
__device__ __forceinline__ void bar_records(const SweepArgs& a, const BarProg& b, int32_t r0, int32_t r1,
                                            const int4 op_first, int lane, Begin begin, Record record, Child child) {
  int e = 0;
  bool fresh = true;
  for (int32_t c = r0; c < r1; c += 32) {
    int4 op = op_first;
    if (r1 - r0 > 32) op = c + lane < r1 ? __ldg(a.bar.ops + c + lane) : make_int4(OP_END, 0, 0, 0);
    int2 rel = make_int2(0, 0);
    int64_t off = 0;
    if (op.x >= 0) {
      rel = __ldcg(a.bar.rel + c + lane);
      if (TL) off = __ldg(a.inst_off + op.x);
    }
    const int n = min(32, r1 - c);
    const unsigned stops = __ballot_sync(kBarFull, op.x < 0);
    for (int i = 0; i < n; ++i) {
      const unsigned after = stops & ~((1u << i) - 1u);
      const int stop = after ? min(__ffs(after) - 1, n) : n;     // records [i, stop) are the engine's
      if (fresh && (i < stop || __shfl_sync(kBarFull, op.x, i) == OP_LOOP)) {
        begin(e);
        fresh = false;
      }
      for (; i < stop; ++i)
        record((uint32_t)__shfl_sync(kBarFull, rel.x, i), (uint32_t)__shfl_sync(kBarFull, rel.y, i),
               TL ? __shfl_sync(kBarFull, off, i) : 0);
      if (i == n) break;
      if (__shfl_sync(kBarFull, op.x, i) == OP_LOOP) {
        child(b.loop_base + (__shfl_sync(kBarFull, op.y, i) - b.le_base) / b.ne,
              (int64_t)(((uint64_t)(uint32_t)__shfl_sync(kBarFull, op.w, i) << 32) |
                        (uint32_t)__shfl_sync(kBarFull, op.z, i)), e);
      } else {                              // the engine's END
        ++e;
        fresh = true;
      }
    }
  }
}

// The instances of iterations gb .. gb + 32 U - 1 (FULL: all below g1) of
// loop l, whose host h has no moving loop in it or before it in its parent's
// body: a lane per iteration, U iterations per lane; toff: l's start in h's
// iteration; op_first: the body's first 32 records.  j0: a row at or before
// the first iteration's, moved on.
template <bool TL, int U, bool FULL>
__device__ __forceinline__ void bar_times(const SweepArgs& a, const BarProg& b, int l, int h, const LoopInfo& H,
                                          uint32_t toff, int32_t r0, int32_t r1, const int4 op_first, int32_t gb,
                                          int32_t g1, int32_t& j0, int lane, unsigned long long& chk) {
  const int32_t* rp = a.rowptr + H.rowptr_off;
  const int32_t* F = a.bar.F + a.bar.bl[H.parent].foff;
  const int2 ko = __ldcg(a.bar.ko + h);
  const bool ok = FULL || gb + lane < g1;                  // U = 1 unless FULL
  const int32_t row_l = bar_row(b, l), row_h = bar_row(b, h);
  uint32_t base[U], a1[U], a2[U];
  int32_t jr[U], dt[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int32_t g = FULL ? gb + 32 * u + lane : min(gb + lane, g1 - 1);
    int32_t lo;
    bar_rows(rp, H.n_parent, gb + 32 * u, g, j0, lane, jr[u], lo);
    j0 = __shfl_sync(kBarFull, jr[u], 31);
    dt[u] = g - lo;
    base[u] = (uint32_t)__ldcg(F + jr[u]) + (uint32_t)ko.y + toff + (uint32_t)ko.x * (uint32_t)dt[u];
  }
  bar_records<TL>(
      a, b, r0, r1, op_first, lane,
      [&](int e) {                          // the engine's position in its stream at the iterations' starts
        const int2 rc = __ldg(a.bar.rowc + row_h + e);
        const uint32_t first = (uint32_t)rc.x + (l != h ? (uint32_t)__ldg(a.bar.rowc + row_l + e).x : 0u);
        const int32_t* Fe = F + (int64_t)(1 + e) * H.n_parent;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t n = (uint32_t)__ldcg(Fe + jr[u]) + first + (uint32_t)rc.y * (uint32_t)dt[u];
          a1[u] = n * kMixA + (uint32_t)e;
          a2[u] = n * kMixB + (uint32_t)e;
        }
      },
      [&](uint32_t di, uint32_t dr, int64_t out) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          a1[u] += kMixA;
          a2[u] += kMixB;
          const uint32_t issue = base[u] + di, retire = base[u] + dr;
          if (ok) {
            chk += inst_mix(issue, retire, a1[u], a2[u]);
            if (TL) {
              a.issue[out + gb + 32 * u + lane] = (int32_t)issue;
              a.retire[out + gb + 32 * u + lane] = (int32_t)retire;
            }
          }
        }
      },
      [&](int c, int64_t, int e) {          // a fixed loop: its time is in rel
        const uint32_t n = (uint32_t)__ldg(a.bar.rowc + bar_row(b, c) + e).y;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          a1[u] += n * kMixA;
          a2[u] += n * kMixB;
        }
      });
}

// The same for any loop, 32 iterations.
template <bool TL>
__device__ __noinline__ unsigned long long bar_times_any(const SweepArgs& a, const BarProg& b, int l, int h, int32_t r0,
                                                         int32_t r1, const int4 op_first, int32_t gb, int32_t g1,
                                                         int lane) {
  const LoopInfo H = a.loop[h];
  const BarLoop B = a.bar.bl[h];
  const bool ok = gb + lane < g1;
  const int32_t g = min(gb + lane, g1 - 1);
  unsigned long long chk = 0;
  int c = l, sib = -1;                      // sib: h's items before l that hold moving loops
  uint32_t toff = 0;
  for (; c != h; c = a.loop[c].parent) {
    toff += (uint32_t)__ldcg(a.bar.ko + c).y;
    if (a.loop[c].parent == h && a.bar.bl[c].esib > 0) sib = a.bar.bl[c].item;
  }
  const int ih = __ldg(a.plan_ptr + h);
  int32_t j = 0, lo = 0;
  const bool climb = H.parent >= 0 && B.foff < 0;
  if (climb) {
    const int32_t* rp = a.rowptr + H.rowptr_off;
    j = bar_row_of(rp, H.n_parent, g);
    lo = __ldg(rp + j);
  }
  auto start = [&](int q) -> uint32_t {
    uint32_t v = climb ? bar_start(a, b, h, H, B, j, lo, g, q)
                 : H.parent < 0 ? 0u : (uint32_t)__ldcg(bar_starts(a, B.foff, H.total, q) + g);
    if (sib >= 0) v += bar_children(a, b, ih, sib, g, q, false);
    return v;
  };
  const uint32_t base0 = start(0) + toff;
  uint32_t base = base0, a1 = 0, a2 = 0;
  bar_records<TL>(
      a, b, r0, r1, op_first, lane,
      [&](int e) {
        const uint32_t n = start(1 + e) + (l != h ? (uint32_t)__ldg(a.bar.rowc + bar_row(b, l) + e).x : 0u);
        base = base0;
        a1 = n * kMixA + (uint32_t)e;
        a2 = n * kMixB + (uint32_t)e;
      },
      [&](uint32_t di, uint32_t dr, int64_t out) {
        a1 += kMixA;
        a2 += kMixB;
        const uint32_t issue = base + di, retire = base + dr;
        if (ok) {
          chk += inst_mix(issue, retire, a1, a2);
          if (TL) {
            a.issue[out + g] = (int32_t)issue;
            a.retire[out + g] = (int32_t)retire;
          }
        }
      },
      [&](int ch, int64_t crp, int e) {     // past a child loop: its instances, and its time unless fixed
        const int32_t x0 = __ldg(a.rowptr + crp + g), x1 = __ldg(a.rowptr + crp + g + 1);
        if (a.bar.bl[ch].host == ch) base += bar_span(a, b, ch, x0, x1, 0);
        const uint32_t n = bar_span(a, b, ch, x0, x1, 1 + e);
        a1 += n * kMixA;
        a2 += n * kMixB;
      });
  return chk;
}

template <int MODE, bool TL, bool FUSED>
__device__ __forceinline__ bool bar_body(const SweepArgs& a, int tile, int l, const BarLoop& B, int32_t* at, int lane,
                                         unsigned long long& chk) {
  const ProgInfo& pi = a.prog[B.prog];
  const BarProg b{pi.le_base, pi.loop_base, pi.ne};
  const int32_t row = bar_row(b, l);
  const int32_t g0 = (tile - B.tile0) * B.iters, g1 = min(a.loop[l].total, g0 + B.iters);
  const int32_t r0 = __ldg(a.bar.op_ptr + row), r1 = __ldg(a.bar.op_ptr + row + b.ne);
  int4 op = r0 + lane < r1 ? __ldg(a.bar.ops + r0 + lane) : make_int4(OP_END, 0, 0, 0);
  const int4 op_first = op;
  bool bad = false;
  for (int32_t c = r0; c < r1; c += 32) {
    if (c > r0) op = c + lane < r1 ? __ldg(a.bar.ops + c + lane) : make_int4(OP_END, 0, 0, 0);
    if (__ballot_sync(kBarFull, op.x >= 0 && op.z > 0)) bad = bar_waits<MODE, FUSED>(a, b, g0, g1, op, at, lane) || bad;
  }
  const int h = B.host;
  const BarLoop BH = a.bar.bl[h];
  int32_t gb = g0;
  if (BH.foff < 0 && BH.esib == 0 && h != b.loop_base) {
    const LoopInfo H = a.loop[h];
    uint32_t toff = 0;
    for (int c = l; c != h; c = a.loop[c].parent) toff += (uint32_t)__ldcg(a.bar.ko + c).y;
    int32_t j0 = bar_row_warp(a.rowptr + H.rowptr_off, H.n_parent, g0, lane);
    for (; gb + 32 * kBarU <= g1; gb += 32 * kBarU)
      bar_times<TL, kBarU, true>(a, b, l, h, H, toff, r0, r1, op_first, gb, g1, j0, lane, chk);
    for (; gb < g1; gb += 32)
      bar_times<TL, 1, false>(a, b, l, h, H, toff, r0, r1, op_first, gb, g1, j0, lane, chk);
  }
  for (; gb < g1; gb += 32) chk += bar_times_any<TL>(a, b, l, h, r0, r1, op_first, gb, g1, lane);
  return __ballot_sync(kBarFull, bad) != 0;
}

__device__ __forceinline__ void bar_add(const SweepArgs& a, int p, unsigned long long chk, int lane) {
  for (int o = 16; o > 0; o >>= 1) chk += __shfl_xor_sync(kBarFull, chk, o);
  if (lane == 0) atomicAdd(a.checksum + p, chk);
}

// One tile in the sweep's launch.  Returns the program when this was its
// last tile and a wait differed (it has to be swept), else -1.
template <int MODE, bool TL, bool FUSED>
__device__ __forceinline__ int bar_tile(const SweepArgs& a, int tile, int32_t* at, int lane) {
  const int l = __ldg(a.bar.tile_loop + tile);
  const BarLoop B = a.bar.bl[l];
  if (__ldcg(a.bar.left + B.prog) < 0) return -1;
  unsigned long long chk = 0;
  const bool bad = bar_body<MODE, TL, FUSED>(a, tile, l, B, at, lane, chk);
  bar_add(a, B.prog, chk, lane);
  __threadfence();                 // the tile's results before its count, for a sweep of the program
  __syncwarp();
  int32_t old = 0;
  if (lane == 0) {
    if (bad) atomicOr(a.bar.left + B.prog, kBarBad);
    old = atomicSub(a.bar.left + B.prog, 1);
    __threadfence();
  }
  old = __shfl_sync(kBarFull, old, 0);
  return old == (kBarBad | 1) ? B.prog : -1;
}

// Waits until every program is planned (a plan waits for nothing, and every
// warp takes its plans before its tiles, so the count is reached); bounded
// all the same: false after about a minute.
__device__ __forceinline__ bool bar_planned(const SweepArgs& a, int lane) {
  int ok = 0;
  if (lane == 0) {
    for (long long n = 0; n < 100000000ll && !ok; ++n) {
      int32_t v;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(a.bar.plans) : "memory");
      ok = v >= a.n_programs;
      if (!ok) __nanosleep(100);
    }
  }
  ok = __shfl_sync(kBarFull, ok, 0);
  return ok != 0;
}

}  // namespace
}  // namespace syncgb
