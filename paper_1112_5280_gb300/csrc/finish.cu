// Reduction totals and scalar finishers of batched launches (k_finish).
//
// A reducing kernel leaves one FP64 partial per tile (per sum, strided by 3) at
// partials[slot.tile0 + tile]. k_finish, issued right after it on the same stream, adds
// each slot's partials in a fixed order (slot_totals in batch.cuh) and runs the slot's scalar
// program (run_fin). The kernel boundary orders the partials. The groups of a slot spread a
// large one over several SMs (one SM adds FP64 at 2 per clock, and a 32^3x64 slot has 16 k
// partials), while a small slot keeps a single CTA and no ticket.
#include "launch.h"

namespace lqcd {
namespace {

constexpr int FINISH_THREADS = FINISH_LANES;

__global__ void __launch_bounds__(FINISH_THREADS) k_finish(const Launch L) {
  pdl_entry();
  const int slot = blockIdx.x, q = blockIdx.y;
  if (slot >= L.nslots) return;
  const Work& w = work_of(L, slot);
  if ((!w.red && w.fin == FIN_NONE) || !slot_runs(w) || q >= finish_groups(w.ntiles)) return;
  double tot[3] = {0, 0, 0};
  const bool done = w.red >= 2 ? slot_totals<FINISH_THREADS, 3>(w, q, L.partials, tot)
                               : slot_totals<FINISH_THREADS, 1>(w, q, L.partials, tot);
  if (done) run_fin(w, tot);
}

}  // namespace

cudaError_t launch_finish(const Launch& L, cudaStream_t s) {
  if (L.nslots <= 0) return cudaSuccess;
  // enough groups for the largest slot (no slot has more tiles than the launch)
  return launch_k(k_finish, dim3(L.nslots, finish_groups(L.ntiles)), dim3(FINISH_THREADS), 0, s, L);
}

}  // namespace lqcd
