// Schedule simulator, program-order sweep: the launchers of the sweep kernel
// (its device code, shared with the piece-parallel launches, is sweep.cuh).
#include "sweep.cuh"

namespace syncgb {
namespace {

template <int MODE, bool BB>
cudaError_t launch3(const SweepArgs& a, size_t smem, int num_sms, cudaStream_t s) {
  long long items = a.n_programs;
  bool spread = true;
  auto run = [&](auto kern) { return run_sweep(kern, a, items, smem, num_sms, s, spread); };
  if constexpr (BB) {
    if (a.bar.on && a.bar.n_tiles > items) items = a.bar.n_tiles;
    if (a.bar.on || a.bar.todo) {
      spread = false;                          // tiles are dealt out kWarps a CTA
      if (a.dep)
        return a.issue ? run(k_sweep<MODE, true, true, true, false, true>) : run(k_sweep<MODE, true, false, true, false, true>);
      return a.issue ? run(k_sweep<MODE, true, true, false, false, true>) : run(k_sweep<MODE, true, false, false, false, true>);
    }
  }
  if (a.dep) return a.issue ? run(k_sweep<MODE, BB, true, true>) : run(k_sweep<MODE, BB, false, true>);
  return a.issue ? run(k_sweep<MODE, BB, true, false>) : run(k_sweep<MODE, BB, false, false>);
}

}  // namespace

size_t sweep_smem_bytes(int sem_cap, int frame_depth, int ring, bool maps) {
  return kWarps * warp_bytes(sem_cap, frame_depth, ring, maps);
}

int sweep_ring_for(int sem_cap, int frame_depth, bool maps, size_t limit) {
  for (int r = kRingMax; r >= 1; r >>= 1)
    if (sweep_smem_bytes(sem_cap, frame_depth, r, maps) <= limit) return r;
  return 0;
}

int sweep_ring(int sem_cap, int frame_depth, bool maps) {
  const int r = maps ? sweep_ring_for(sem_cap, frame_depth, maps, 108 * 1024) : 0;
  return r ? r : sweep_ring_for(sem_cap, frame_depth, maps, 200 * 1024);
}

// The maps' kernel runs 16 warps per SM, the walk's 24, or fewer where the
// rings are large.  A sweep's time is taken as the longest item's and all
// items' over the warps an SM runs at full rate (15.5, 10.7 or 6.9 walked with
// 3, 2 or 1 CTAs, 8.8 or 6.3 by maps with 2 or 1), added as squares; the maps
// have to promise 9%, or 5% where the longest item makes the time.  Walked / by
// maps, us, one loop of 16 records and trips of 64: 500 programs 557 / 209,
// 3000 829 / 564, 20000 4240 / 2640; 12 records without waits inside an
// iteration, trips of 19, 3000 296 / 424; 4 records, trips of 32, 3000 236 / 359; 16 records, trips
// of 8, 500 683 / 545, 3000 1027 / 1437; trips of 16, 3000 923 / 855, with 36
// waited semaphores 923 / 1125, with 120 1954 / 1129; 40 records (no map),
// 3000 15240 / 28570; two loops in turn (the warp keeps one map), 3000 6370 /
// 9090; a loop entered once (never mapped), 3000 46 / 56; chain 777 9220 /
// 6190, 4864 12600 / 9490; depth2 4096 4890 / 1150; sync-bound 65536 33960 /
// 12510; branching trees 6000 844 / 1417.  Of many items the longest no longer
// decide, and the estimate is good for loops of one size only: past 80 an SM
// they need 320 instances a statement as well (chain 264, 16384 14.5 / 14.7
// ms, 32768 16.4 / 21.3; depth2 540, 16384 7.0 / 4.3).
bool sweep_maps(const SweepCost& c, int num_sms, int sem_cap, int frame_depth) {
  const int ring_m = sweep_ring(sem_cap, frame_depth, true), ring_w = sweep_ring(sem_cap, frame_depth, false);
  if (ring_m == 0) return false;
  const auto ctas = [&](int ring, bool maps) {       // resident per SM, a kilobyte of which is the system's
    return (int)(228 * 1024 / (sweep_smem_bytes(sem_cap, frame_depth, ring, maps) + 1024));
  };
  const int walked = ctas(ring_w, false), mapped = ctas(ring_m, true);
  const double w = (double)c.walk / ((walked >= 3 ? 15.5 : walked == 2 ? 10.7 : 6.9) * num_sms);
  const double m = (double)c.map / ((mapped >= 2 ? 8.8 : 6.3) * num_sms);
  const double lw = (double)c.walk_max, lm = (double)c.map_max;
  const double most = m < lm / 2 ? 0.95 : 0.91;
  return lm * lm + m * m < most * most * (lw * lw + w * w) &&
         (c.items <= 80 * num_sms || c.n_inst >= 320 * c.n_stmt[0] || c.n_stmt[1] >= 4 * c.n_stmt[0]);
}

cudaError_t launch_sweep(const SweepArgs& a, bool barrier, int num_sms, cudaStream_t s) {
  if (a.n_programs == 0) return cudaSuccess;
  if (a.ring < 1) return cudaErrorInvalidConfiguration;
  if (a.maps) return launch_sweep_maps(a, num_sms, s);
  const size_t smem = sweep_smem_bytes(a.sem_cap, a.frame_depth, a.ring, false);
  if (a.mode == SYNC_THR_PERLOOP)
    return barrier ? launch3<SYNC_THR_PERLOOP, true>(a, smem, num_sms, s)
                   : launch3<SYNC_THR_PERLOOP, false>(a, smem, num_sms, s);
  if (a.mode == SYNC_THR_PERENGINE)
    return barrier ? launch3<SYNC_THR_PERENGINE, true>(a, smem, num_sms, s)
                   : launch3<SYNC_THR_PERENGINE, false>(a, smem, num_sms, s);
  return barrier ? launch3<SYNC_THR_COUNT, true>(a, smem, num_sms, s)
                 : launch3<SYNC_THR_COUNT, false>(a, smem, num_sms, s);
}

}  // namespace syncgb
