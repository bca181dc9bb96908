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
