// Barrier scheme by intervals (bar.cuh): the launches of a batch with split
// programs, whose loops are scheduled by separate warps instead of one warp
// per program.
#include "bar.cuh"

namespace syncgb {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t warp_id() { return (blockIdx.x * (int64_t)kThreads + threadIdx.x) >> 5; }

// Program p is left to the sweep (listed once).
__device__ __forceinline__ void leave(const SweepArgs& a, int32_t* todo, int p) { todo[1 + atomicAdd(todo, 1)] = p; }

template <int MODE, bool FUSED>
__global__ void __launch_bounds__(kThreads) k_bar_classes(const __grid_constant__ SweepArgs a, int32_t* todo) {
  const int64_t p = warp_id();
  const int lane = threadIdx.x & 31;
  if (p >= a.n_programs) return;
  const ProgInfo pi = a.prog[p];
  bar_counts(a, (int)p, pi, lane);
  const bool ok = bar_in_time<MODE>(a, pi) && bar_classes<MODE, FUSED>(a, pi, lane);
  if (lane == 0) {
    a.bar.left[p] = ok ? 1 : -1;
    if (!ok) leave(a, todo, (int)p);
  }
}

__global__ void __launch_bounds__(kThreads) k_bar_schedule(const __grid_constant__ SweepArgs a, int32_t* todo,
                                                          int32_t n_loops) {
  __shared__ int32_t at[kThreads];
  const int64_t l = warp_id();
  const int lane = threadIdx.x & 31;
  if (l >= n_loops || a.bar.bl[l].host != l) return;
  const int p = a.bar.bl[l].prog;
  if (__ldcg(a.bar.left + p) < 0 || a.loop[l].total == 0) return;
  if (!bar_schedules(a, a.prog[p], (int)l, at + (threadIdx.x & ~31), lane) && lane == 0)
    if (atomicExch(a.bar.left + p, -1) >= 0) leave(a, todo, p);
}

__global__ void __launch_bounds__(kThreads) k_bar_compose(const __grid_constant__ SweepArgs a) {
  const int64_t p = warp_id();
  if (p >= a.n_programs || a.bar.left[p] < 0) return;
  bar_compose(a, (int)p, a.prog[p], threadIdx.x & 31);
}

template <int MODE, bool TL, bool FUSED>
__global__ void __launch_bounds__(kThreads, 3) k_bar_tiles(const __grid_constant__ SweepArgs a, int32_t* todo) {
  __shared__ int32_t at[kThreads];
  const int64_t tile = warp_id();
  const int lane = threadIdx.x & 31;
  if (tile >= a.bar.n_tiles) return;
  const int l = __ldg(a.bar.tile_loop + tile);
  const BarLoop B = a.bar.bl[l];
  if (__ldcg(a.bar.left + B.prog) < 0) return;
  unsigned long long chk = 0;
  const bool bad = bar_body<MODE, TL, FUSED>(a, (int)tile, l, B, at + (threadIdx.x & ~31), lane, chk);
  bar_add(a, B.prog, chk, lane);
  if (bad && lane == 0 && !(atomicOr(a.bar.left + B.prog, kBarBad) & kBarBad)) leave(a, todo, B.prog);
}

int blocks(int64_t warps) { return (int)((warps * 32 + kThreads - 1) / kThreads); }

template <int MODE, bool FUSED>
cudaError_t intervals(const SweepArgs& a, int32_t* todo, int32_t n_loops, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(todo, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  k_bar_classes<MODE, FUSED><<<blocks(a.n_programs), kThreads, 0, s>>>(a, todo);
  if ((e = launched()) != cudaSuccess) return e;
  k_bar_schedule<<<blocks(n_loops), kThreads, 0, s>>>(a, todo, n_loops);
  if ((e = launched()) != cudaSuccess) return e;
  k_bar_compose<<<blocks(a.n_programs), kThreads, 0, s>>>(a);
  if ((e = launched()) != cudaSuccess) return e;
  const int grid = blocks(a.bar.n_tiles < 1 ? 1 : a.bar.n_tiles);
  if (a.issue) k_bar_tiles<MODE, true, FUSED><<<grid, kThreads, 0, s>>>(a, todo);
  else k_bar_tiles<MODE, false, FUSED><<<grid, kThreads, 0, s>>>(a, todo);
  return launched();
}

}  // namespace

cudaError_t launch_intervals(const SweepArgs& a, int32_t* todo, int32_t n_loops, cudaStream_t s) {
  if (a.n_programs == 0) return cudaSuccess;
  if (a.mode == SYNC_THR_PERLOOP)
    return a.dep ? intervals<SYNC_THR_PERLOOP, true>(a, todo, n_loops, s) : intervals<SYNC_THR_PERLOOP, false>(a, todo, n_loops, s);
  if (a.mode == SYNC_THR_PERENGINE)
    return a.dep ? intervals<SYNC_THR_PERENGINE, true>(a, todo, n_loops, s) : intervals<SYNC_THR_PERENGINE, false>(a, todo, n_loops, s);
  return a.dep ? intervals<SYNC_THR_COUNT, true>(a, todo, n_loops, s) : intervals<SYNC_THR_COUNT, false>(a, todo, n_loops, s);
}

}  // namespace syncgb
