// Barrier-free sweep: the iterations of a loop's trip by its max-plus map,
// for loops whose iterations are one straight line of at most 32 records: no
// child loops but fixed ones (which run exactly once on every visit, so
// their records' instances are the loop's iterations and they cost every
// engine the same each time), and no barrier-fallback barrier, which joins
// the engines and is no record.
//
// With its waits inside an iteration fixed, every issue and retire of an iteration is a
// maximum, over the engines' cursors and last retires at its start and the
// times its waits on earlier increments are satisfied (the map's inputs), of
// that value plus a sum of costs along a path (all costs >= 0, no constant
// terms).  The weights depend on the loop alone: they are read off once by
// relaxing the body with one input at 0 and the others at none.  A trip then
// takes two phases:
//   the inputs of the next iteration from this one's, a lane per input (its
//     cursor or last retire is the last record's, a loop-carried wait its
//     producer's retire k iterations back, an outer wait constant): the only
//     serial part, about 2 instructions per input and iteration;
//   all instances of up to 32 iterations at once, a lane per iteration, a
//     record at a time: 2 instructions per input and record, 14 for the
//     checksum.
// It holds for a trip whose thresholds name the producers the dependencies
// do, in every iteration (compared first); any other trip is walked.  What
// bounds it is one warp's dependent instructions: an iteration of 17 records
// took 1500 cycles walked; with 11 inputs phase 1 takes 119, phase 2 184 per
// record and 32 iterations, the comparison 565 to 1100 a batch.  Barrier-free,
// walked / by maps: 4096 depth-2 programs 4.9 / 1.1 ms, 777 chain programs
// 9.2 / 6.2, 256 attention programs (pieces) 14.9 / 7.9, 65536 sync-bound
// ones 34.0 / 12.5.  Two records per half warp for short trips, skipping a
// record's groups without weights, and unrolling by 4 were no faster.
#pragma once

namespace syncgb {
namespace {

constexpr int32_t kTripNone = -(1 << 30);
constexpr int kTripRow = kTripCols + 1;     // odd: a lane per row without bank conflicts
// the warp's ints (kTripInts)
constexpr int kTripIn = 2 * 32 * kTripCols;         // [32][kTripRow] inputs per iteration
constexpr int kTripSeg = kTripIn + 32 * kTripRow;   // [32] int64: a dependency's thresholds
constexpr int kTripDep = kTripSeg + 64;             // [32] kind | k << 2 | rank << 4 | increments << 10 | semaphore << 16 | S in the body << 31
constexpr int kTripCol = kTripDep + 32;             // [32] kind | lane << 4 | dependency << 12 | k << 20 | engine << 24
constexpr int kTripRec = kTripCol + 32;             // [32] engine | records of it << 8 | rank among them << 16
constexpr int kTripInc = kTripRec + 32;             // [32] semaphore | rank << 16 | increments << 24, or -1
constexpr int kTripOut = kTripInc + 32;             // [32] int4 x 2: a record's outputs in this trip (see trip_times)
constexpr int kTripR = kTripOut + 8 * 32;           // [32] a dependency's consumer-grouped index
constexpr int kTripX = kTripR + 32;                 // [32] a record's global instruction
constexpr int kTripTail = kTripX + 32;              // [32] an engine's control costs after its last record (all, without one)
constexpr int kTripHead = kTripTail + 32;           // {loop, inputs (0: none yet), dependencies | records << 8,
                                                    //  iterations walked (< 0: never), maps allowed}
static_assert(kTripHead + 16 == kTripInts, "trip map layout");
enum : int { TD_CHUNK = 0, TD_CARRIED = 1, TD_OUTER = 2 };                       // dependencies
enum : int { TC_CURSOR = 0, TC_RETIRE = 1, TC_CARRIED = 2, TC_OUTER = 3, TC_NONE = 4 };   // inputs

// An engine's records in one iteration of a loop, fixed loops entered: f(op
// record's index, record, the control costs since the engine's previous one);
// returns the costs after the last.
template <int MODE, class F>
__device__ __forceinline__ int32_t trip_walk(const SweepArgs& a, const BarProg& b, int row, int e, F f) {
  const bool elide = a.prm.trip_register_elision != 0;
  int back[SYNC_MAX_DEPTH + 1];
  int d = 0;
  int32_t pre = 0;
  for (int i = __ldg(a.bar.op_ptr + row + e);;) {
    const int4 o = __ldg(a.bar.ops + i);
    if (o.x >= 0) {
      f(i, o, pre);
      pre = 0;
      ++i;
    } else if (o.x == OP_LOOP) {
      const int c = b.loop_base + (o.y - b.le_base) / b.ne;
      const int32_t reg = elide && __ldg(a.lflag + c) ? 0 : a.prm.c_regop;       // r-hat := 0, r-hat++
      pre += 2 * reg + a.prm.c_regop + a.prm.c_branch + hoist_ops<MODE, false>(a, o.y + e);
      back[d++] = i + 1;
      i = __ldg(a.bar.op_ptr + o.y + e);
    } else {
      if (d == 0) return pre;
      i = back[--d];
    }
  }
}

// Builds the map of a loop.  False: never (too many records, inputs or
// dependencies, a far offset, a cycle of waits).
template <int MODE>
__device__ __noinline__ bool trip_build(const SweepArgs& a, int32_t* map, const BarProg b, int loop, int lane) {
  const int ne = b.ne, row = bar_row(b, loop);
  // the records, engine by engine
  int32_t *ids = map + kTripIn, *pres = ids + 32, *engs = ids + 64, *sem_of = ids + 96;
  int cnt = 0;
  int32_t tail = 0;
  if (lane < ne) tail = trip_walk<MODE>(a, b, row, lane, [&](int, const int4&, int32_t) { ++cnt; });
  int at = cnt;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, at, o);
    if (lane >= o) at += v;
  }
  const int n_rec = __shfl_sync(kFull, at, 31);
  if (n_rec == 0 || n_rec > 32) return false;
  at -= cnt;
  const int first_of = at;
  if (lane < ne)
    trip_walk<MODE>(a, b, row, lane, [&](int i, const int4&, int32_t pre) {
      ids[at] = i;
      pres[at] = pre;
      engs[at++] = lane;
    });
  map[kTripTail + lane] = tail;
  __syncwarp();
  const bool have = lane < n_rec;
  const int op = have ? ids[lane] : -1, e = have ? engs[lane] : 0;
  const int head = __shfl_sync(kFull, first_of, e);
  const int4 rec = have ? __ldg(a.bar.ops + op) : make_int4(0, 0, 0, 0);
  const int4 sr = have ? __ldg(a.opsem + op) : make_int4(-1, 0, 0, 0);
  const int32_t ii = a.prm.ii, lat = rec.y;
  const int32_t A = have ? pres[lane] + wait_ops<MODE>(a, rec, sr.w) + ii : 0;
  const int32_t sem = sr.x;
  map[kTripX + lane] = rec.x;
  sem_of[lane] = sem;
  // engine runs and semaphore groups
  const unsigned run = __match_any_sync(kFull, have ? e : 32 + lane), grp = __match_any_sync(kFull, sem >= 0 ? sem : -2 - lane);
  map[kTripRec + lane] = e | __popc(run) << 8 | __popc(run & lanemask_le()) << 16;
  map[kTripInc + lane] = sem >= 0 ? sem | __popc(grp & lanemask_le()) << 16 | __popc(grp) << 24 : -1;
  __syncwarp();
  // dependencies, one index each
  const int z = rec.z;
  int pre = z;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, pre, o);
    if (lane >= o) pre += v;
  }
  const int nd = __shfl_sync(kFull, pre, 31);
  pre -= z;
  if (nd > 32 || __ballot_sync(kFull, sem > 0x7fff)) return false;
  bool ok = true;
  uint64_t intra = 0;
  int n_intra = 0;
  for (int j = 0; j < z; ++j) {
    const int r = rec.w + j;
    const DepInfo D = a.bar.dep[__ldg(a.bar.ddep + r)];
    const BarDep bd = a.bar.bdep[r];
    const int32_t s = __ldg(a.dsem + r);
    int kind = TD_OUTER, k = 0, rank = 0, inc = 0, p = 0;
    if (s < 0 || s > 0x7fff) { ok = false; continue; }
    int sl = bd.cons_loop;                  // the common loop S
    for (int u = 0; u < D.up; ++u) sl = a.loop[sl].parent;
    const bool body = a.bar.bl[sl].host == loop;
    // carried at a fixed loop: no wait (one iteration a trip)
    if (body && (D.k == 0 || sl == loop)) {
      while (p < n_rec && ids[p] != bd.prod_op) ++p;
      k = D.k;
      if (p == n_rec || k > 3) { ok = false; continue; }
      kind = k == 0 ? TD_CHUNK : TD_CARRIED;
      for (int i = 0; i < n_rec; ++i)
        if (sem_of[i] == s) { ++inc; rank += i <= p; }
      if (kind == TD_CHUNK) {
        if (n_intra == kMaxIntra) { ok = false; continue; }
        intra |= (uint64_t)p << (5 * n_intra++);
      }
    }
    reinterpret_cast<int64_t*>(map + kTripSeg)[pre + j] = __ldg(a.dseg + r);
    map[kTripR + pre + j] = r;
    map[kTripDep + pre + j] = kind | k << 2 | rank << 4 | inc << 10 | s << 16 | (body ? 1 << 31 : 0);
    map[kTripCol + pre + j] = lane | p << 8;       // until the columns are known
  }
  if (__ballot_sync(kFull, !ok)) return false;
  __syncwarp();
  const int32_t dep_of = lane < nd ? map[kTripDep + lane] : TD_CHUNK, lanes_of = map[kTripCol + lane];
  __syncwarp();
  const unsigned ext = __ballot_sync(kFull, lane < nd && (dep_of & 3) != TD_CHUNK);
  const int deepest = (int)__reduce_max_sync(kFull, (unsigned)n_intra);
  map[kTripCol + lane] = TC_NONE;
  int2* w = reinterpret_cast<int2*>(map);
  for (int c = 0; c < kTripCols; ++c) w[lane * kTripCols + c] = make_int2(kTripNone, kTripNone);
  __syncwarp();
  int col = 0;
  for (int q = 0; q < 2 * ne + 32; ++q) {
    const int kind = q < ne ? TC_CURSOR : q < 2 * ne ? TC_RETIRE : TC_CARRIED;
    const int at = kind == TC_CURSOR ? q : kind == TC_RETIRE ? q - ne : q - 2 * ne;
    int to = 0, info = 0;
    if (kind == TC_CARRIED) {
      if (!((ext >> at) & 1)) continue;
      const int d = __shfl_sync(kFull, dep_of, at), l = __shfl_sync(kFull, lanes_of, at);
      to = l & 255;
      info = ((d & 3) == TD_OUTER ? TC_OUTER : TC_CARRIED) | (l >> 8) << 4 | at << 12 | ((d >> 2) & 3) << 20;
    } else {
      const unsigned of = __ballot_sync(kFull, have && e == at);
      if (!of) continue;
      info = kind | (31 - __clz(of)) << 4 | at << 24;
    }
    if (col == kTripCols) return false;
    const int32_t t_in = kind == TC_CURSOR && e == at ? 0 : kTripNone, lr = kind == TC_RETIRE && e == at ? 0 : kTripNone;
    const int32_t known = kind == TC_CARRIED && lane == to ? 0 : kTripNone;
    int32_t r_intra = kTripNone, issue = kTripNone, retire = kTripNone;
    bool settled = false;
    for (int pass = 0; pass < n_rec + 2 && !settled; ++pass) {
      const int32_t ready = max(known, r_intra);
      int32_t Ai = A, Bi = have && ready >= 0 ? ready + ii : kTripNone;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t Ap = __shfl_up_sync(kFull, Ai, o), Bp = __shfl_up_sync(kFull, Bi, o);
        if (lane - o >= head) { Bi = max(Bp + Ai, Bi); Ai += Ap; }
      }
      issue = max(t_in + Ai, Bi) - ii;
      if (issue < 0 || !have) issue = kTripNone;
      int32_t rv = issue >= 0 ? issue + lat : kTripNone;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t vp = __shfl_up_sync(kFull, rv, o);
        if (lane - o >= head) rv = max(rv, vp);
      }
      retire = have ? max(lr, rv) : kTripNone;
      int32_t nr = kTripNone;
      for (int i = 0; i < deepest; ++i) {
        const int32_t v = __shfl_sync(kFull, retire, (int)(intra >> (5 * i)) & 31);
        if (i < n_intra) nr = max(nr, v);
      }
      settled = !__ballot_sync(kFull, nr >= 0 && nr > issue);
      r_intra = nr;
    }
    if (!settled) return false;
    w[lane * kTripCols + col] = make_int2(issue, retire);
    if (lane == 0) map[kTripCol + col] = info;
    ++col;
  }
  if (lane == 0) {
    map[kTripHead + 1] = col;
    map[kTripHead + 2] = nd | n_rec << 8;
  }
  __syncwarp();
  return true;
}

// Phase 1: the inputs of iterations 0 .. nb-1 into rows, from this lane's
// `in` (moved on past them); G: groups of 4 inputs.  from: the record whose
// issue (a cursor) or retire the input is; h1, h2: a carried input's
// producer one and two iterations back; add: what a cursor gains after it.
template <int G>
__device__ __forceinline__ void trip_inputs(int32_t* map, int lane, int kind, int from, int k, int32_t add, int nb,
                                            int32_t& in, int32_t& h1, int32_t& h2) {
  int32_t rw[4 * G];
  const int2* w = reinterpret_cast<const int2*>(map) + from * kTripCols;
#pragma unroll
  for (int c = 0; c < 4 * G; ++c) {
    const int2 v = w[c];
    rw[c] = kind == TC_CURSOR ? v.x + add : v.y;
  }
  int32_t* row = map + kTripIn + (lane < kTripCols ? lane : kTripCols);
  const bool moves = kind == TC_CURSOR || kind == TC_RETIRE || (kind == TC_CARRIED && k == 1);
  const bool late = __ballot_sync(kFull, kind == TC_CARRIED && k > 1) != 0;
  for (int i = 0; i < nb; ++i) {
    row[i * kTripRow] = in;
    int32_t v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __shfl_sync(kFull, in, q) + rw[q];
#pragma unroll
    for (int c = 4; c < 4 * G; ++c) v[c & 3] = max(v[c & 3], __shfl_sync(kFull, in, c) + rw[c]);
    const int32_t m = max(max(v[0], v[1]), max(v[2], v[3]));
    if (moves) in = m;
    if (late) {
      if (kind == TC_CARRIED && k > 1) in = k == 2 ? h1 : h2;
      h2 = h1;
      h1 = m;
    }
  }
}

// Phase 2: the instances of iterations 0 .. nb-1 (the trip's j0 ..), a lane
// per iteration.  Per record, kTripOut: {history address of its increment in
// the trip's iteration 0 (64 bits), that increment, increments per iteration
// | its rank among them << 8 | semaphore << 16 (-1: nothing waits on it)} and {its position in its
// engine's stream in iteration 0, records of its engine, engine, instruction}.
template <int G, bool TL>
__device__ __forceinline__ void trip_times(const SweepArgs& a, const WarpSmem& S, const int32_t* map, int n_rec,
                                           int lane, int32_t j0, int32_t nb, int32_t lo, unsigned long long& chk) {
  int32_t x[4 * G];
  const int32_t* row = map + kTripIn + lane * kTripRow;
#pragma unroll
  for (int c = 0; c < 4 * G; ++c) x[c] = row[c];
  const int4* out = reinterpret_cast<const int4*>(map + kTripOut);
  const int4* w = reinterpret_cast<const int4*>(map);
  const bool ok = lane < nb;
  const int32_t j = j0 + lane;
#pragma unroll 2
  for (int r = 0; r < n_rec; ++r) {
    const int4 P = out[2 * r], Q = out[2 * r + 1];
    int32_t is[2], re[2];
#pragma unroll
    for (int c = 0; c < 4 * G; c += 2) {
      const int4 p = w[r * (kTripCols / 2) + c / 2];
      if (c == 0) {
        is[0] = x[0] + p.x; re[0] = x[0] + p.y; is[1] = x[1] + p.z; re[1] = x[1] + p.w;
      } else {
        is[0] = max(is[0], x[c] + p.x); re[0] = max(re[0], x[c] + p.y);
        is[1] = max(is[1], x[c + 1] + p.z); re[1] = max(re[1], x[c + 1] + p.w);
      }
    }
    const int32_t issue = max(is[0], is[1]), retire = max(re[0], re[1]);
    const uint32_t nj = (uint32_t)(Q.x + j * Q.y);
    const unsigned long long m =
        inst_mix((uint32_t)issue, (uint32_t)retire, nj * kMixA + (uint32_t)Q.z, nj * kMixB + (uint32_t)Q.z);
    if (ok) chk += m;
    if (TL && ok) tl_write(a, S, __ldg(a.inst_off + Q.w) + lo + j, issue, retire, nj);
    const int32_t per = P.w & 255, n = P.z + j * per;
    if (ok && P.w >= 0) {
      int32_t* h = reinterpret_cast<int32_t*>((uint64_t)(uint32_t)P.y << 32 | (uint32_t)P.x) + j * per;
      *h = retire;
      // of the batch's increments the ring keeps its own number, the last ones
      if ((j0 + nb - j) * per - ((P.w >> 8) & 255) <= S.rmask)
        S.ring[(P.w >> 16) * (S.rmask + 1) + ((n - 1) & S.rmask)] = retire;
    }
  }
}

// Iterations lo .. hi-1 of loop `loop` by its map; the first iteration start
// has been charged.  Returns the first iteration it did not take (the state
// is then as that iteration starts).  FUSED: the thresholds are computed
// (walk level lc), and compared with the Eq. (1) minimum if asked; a trip
// where they differ is walked, which tallies.
template <int MODE, bool TL, bool FUSED>
__device__ __forceinline__ int32_t run_trip(const SweepArgs& a, const WarpSmem& S, const ProgInfo& pi, int loop,
                                            int32_t lo, int32_t hi, int lane, int lc, int32_t iter_cost,
                                            unsigned long long& chk) {
  int32_t* map = S.map;
  const int32_t total = hi - lo;
  if (total < kTripMin || !map[kTripHead + 4]) return lo;
  const int4 hd = *reinterpret_cast<const int4*>(map + kTripHead);
  const bool same = hd.x == loop;
  const int32_t walked = same ? hd.w : 0;
  if (walked < 0 || (!same && (a.bar.bl[loop].foff >= 0 || a.bar.bl[loop].fbar))) return lo;
  int nc = hd.y, nd = hd.z & 255, n_rec = hd.z >> 8;
  if (!same || nc == 0) {
    __syncwarp();
    if (lane == 0) *reinterpret_cast<int4*>(map + kTripHead) = make_int4(loop, 0, 0, walked + total);
    __syncwarp();
    if (walked < kTripLearn) return lo;
    if (!trip_build<MODE>(a, map, bar_prog(pi), loop, lane)) {
      __syncwarp();
      if (lane == 0) *reinterpret_cast<int4*>(map + kTripHead) = make_int4(loop, 0, 0, -1);
      __syncwarp();
      return lo;
    }
    nc = map[kTripHead + 1];
    nd = map[kTripHead + 2] & 255;
    n_rec = map[kTripHead + 2] >> 8;
  }
  // the thresholds name the dependencies' own producers: lane d holds
  // dependency d's {segment, first value, step, iterations without}
  const int64_t* segs = reinterpret_cast<const int64_t*>(map + kTripSeg);
  int64_t seg = 0;
  int32_t T0 = 0, step = 0;
  int dk = 0;
  bool bad = false;
  if (lane < nd) {
    const int32_t D = map[kTripDep + lane];
    seg = segs[lane] + lo;
    const int32_t pub = S.semv[(D >> 16) & 0x7fff];
    dk = (D >> 2) & 3;
    if ((D & 3) == TD_OUTER) {
      if (FUSED) {
        // (carried at a fixed loop of the body: no wait)
        const int r = map[kTripR + lane];
        const DepInfo F = a.dep[__ldg(a.ddep + r)];
        const int below = a.loop[a.bar.bdep[r].cons_loop].depth - a.loop[loop].depth;   // the consumer's loop
        const int2 v = D < 0 ? make_int2(lo, lo) : S.lvl[lc + below - F.up];
        T0 = wait_value(a, F, v.x, v.y, MODE);
        bad = a.chk_counts && minimum(a, F, v.x, v.y, MODE) != T0;
      } else {
        T0 = __ldg(a.thr + seg);
      }
      bad = bad || T0 > pub;
    } else {
      step = (D >> 10) & 63;
      T0 = pub + ((D >> 4) & 63) - dk * step;
    }
  }
  // this lane's input
  const int info = map[kTripCol + lane], kind = info & 15, from = (info >> 4) & 31;
  const int k = (info >> 20) & 3, eng = (info >> 24) & 31, dep = (info >> 12) & 31;
  const int32_t ic = __shfl_sync(kFull, iter_cost, eng), To = __shfl_sync(kFull, T0, dep);
  if (__ballot_sync(kFull, bad)) return lo;
  int32_t in = kTripNone;
  if (kind == TC_CURSOR) in = S.t[eng];
  if (kind == TC_RETIRE) in = S.lr[eng];
  if (kind == TC_OUTER && To > 0) {
    const int s = (map[kTripDep + dep] >> 16) & 0x7fff;
    in = S.semv[s] - To <= S.rmask ? S.ring[s * (S.rmask + 1) + ((To - 1) & S.rmask)] : a.hist[S.semhb[s] + (To - 1)];
  }
  int32_t h1 = kTripNone, h2 = kTripNone;
  // this lane's record
  const int rec = map[kTripRec + lane], inc = map[kTripInc + lane];
  int32_t own_pub = 0;
  if (lane < n_rec) {
    int4 P = make_int4(0, 0, 0, -1);
    if (inc >= 0) {
      const int s = inc & 0xffff;
      own_pub = S.semv[s];
      const int32_t n0 = own_pub + ((inc >> 16) & 255);
      const uint64_t h = reinterpret_cast<uint64_t>(a.hist + S.semhb[s] + (n0 - 1));
      P = make_int4((int32_t)(uint32_t)h, (int32_t)(h >> 32), n0, inc >> 24 | ((inc >> 16) & 255) << 8 | s << 16);
    }
    int4* out = reinterpret_cast<int4*>(map + kTripOut) + 2 * lane;
    out[0] = P;
    out[1] = make_int4(S.nn[rec & 255] + (rec >> 16), (rec >> 8) & 255, rec & 255, map[kTripX + lane]);
  }
  __syncwarp();
  if (FUSED) {                              // all iterations first: the walk cannot take over in a trip
    for (int d = 0; d < nd; ++d) {
      if ((map[kTripDep + d] & 3) == TD_OUTER) continue;    // constant over the trip
      const DepInfo F = a.dep[__ldg(a.ddep + map[kTripR + d])];
      const int32_t w0 = __shfl_sync(kFull, T0, d), st = __shfl_sync(kFull, step, d);
      for (int32_t j = lane; j < total; j += 32) {
        // offset 0 may be carried by a fixed loop: the trip's start is then no matter
        const int32_t T = wait_value(a, F, lo + j, lo, MODE);
        bad = bad || T != (j < F.k ? 0 : w0 + j * st) || (a.chk_counts && minimum(a, F, lo + j, lo, MODE) != T);
      }
    }
    if (__ballot_sync(kFull, bad)) return lo;
  }
  const int groups = (nc + 3) >> 2;
  int32_t done = 0;
  for (; done < total; done += 32) {
    const int32_t nb = min(32, total - done), j = done + lane;
    for (int d = 0; !FUSED && d < nd; d += 4) {
      int32_t T[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t s = __shfl_sync(kFull, seg, min(d + u, nd - 1));
        T[u] = lane < nb ? __ldg(a.thr + s + j) : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = min(d + u, nd - 1);
        const int32_t w0 = __shfl_sync(kFull, T0, q), st = __shfl_sync(kFull, step, q);
        const int kq = __shfl_sync(kFull, dk, q);
        bad = bad || (lane < nb && T[u] != (j < kq ? 0 : w0 + j * st));
      }
    }
    if (__ballot_sync(kFull, bad)) break;
    const int32_t add = a.prm.ii + ic + map[kTripTail + eng];
    if (groups <= 2) trip_inputs<2>(map, lane, kind, from, k, add, nb, in, h1, h2);
    else if (groups == 3) trip_inputs<3>(map, lane, kind, from, k, add, nb, in, h1, h2);
    else if (groups == 4) trip_inputs<4>(map, lane, kind, from, k, add, nb, in, h1, h2);
    else trip_inputs<6>(map, lane, kind, from, k, add, nb, in, h1, h2);
    __syncwarp();
    if (groups <= 2) trip_times<2, TL>(a, S, map, n_rec, lane, done, nb, lo, chk);
    else if (groups == 3) trip_times<3, TL>(a, S, map, n_rec, lane, done, nb, lo, chk);
    else if (groups == 4) trip_times<4, TL>(a, S, map, n_rec, lane, done, nb, lo, chk);
    else trip_times<6, TL>(a, S, map, n_rec, lane, done, nb, lo, chk);
    __syncwarp();
  }
  done = min(done, total);
  if (done == 0) return lo;
  // the engines and semaphores after it
  const unsigned in_body = __reduce_or_sync(kFull, kind == TC_CURSOR ? 1u << eng : 0u);
  if (kind == TC_CURSOR) S.t[eng] = done == total ? in - ic : in;
  if (kind == TC_RETIRE) S.lr[eng] = in;
  if (lane < pi.ne && !((in_body >> lane) & 1)) 
    S.t[lane] += (done == total ? done - 1 : done) * iter_cost + done * map[kTripTail + lane];
  if (lane < n_rec) {
    const int cnt = (rec >> 8) & 255, per = inc >> 24;
    if ((rec >> 16) == cnt) S.nn[rec & 255] += done * cnt;
    if (inc >= 0 && ((inc >> 16) & 255) == per) S.semv[inc & 0xffff] = own_pub + done * per;
  }
  __syncwarp();
  return lo + done;
}

}  // namespace
}  // namespace syncgb
