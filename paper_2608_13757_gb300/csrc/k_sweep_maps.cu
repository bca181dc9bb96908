// Schedule simulator, program-order sweep, barrier-free, trips by their maps
// (trip.cuh): the launcher for the batches that sweep_maps() sends here.
#include "sweep.cuh"

namespace syncgb {
namespace {

template <int MODE>
cudaError_t launch2(const SweepArgs& a, size_t smem, int num_sms, cudaStream_t s) {
  auto run = [&](auto kern) { return run_sweep(kern, a, a.n_programs, smem, num_sms, s); };
  if (a.dep)
    return a.issue ? run(k_sweep<MODE, false, true, true, false, false, true>)
                   : run(k_sweep<MODE, false, false, true, false, false, true>);
  return a.issue ? run(k_sweep<MODE, false, true, false, false, false, true>)
                 : run(k_sweep<MODE, false, false, false, false, false, true>);
}

}  // namespace

cudaError_t launch_sweep_maps(const SweepArgs& a, int num_sms, cudaStream_t s) {
  const size_t smem = sweep_smem_bytes(a.sem_cap, a.frame_depth, a.ring, true);
  if (a.mode == SYNC_THR_PERLOOP) return launch2<SYNC_THR_PERLOOP>(a, smem, num_sms, s);
  if (a.mode == SYNC_THR_PERENGINE) return launch2<SYNC_THR_PERENGINE>(a, smem, num_sms, s);
  return launch2<SYNC_THR_COUNT>(a, smem, num_sms, s);
}

}  // namespace syncgb
