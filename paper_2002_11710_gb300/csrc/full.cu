// The single-instance search with the full evaluation, and the evaluation of one schedule's moves.
#include "search.cuh"
#include "kernels.h"

namespace {

template <bool PEN, bool DL, bool DEBUG, bool BIG>
__global__ void __launch_bounds__(kMaxThreads, 1) tabu_kernel(const __grid_constant__ KParams P) {
  const int C = P.cluster;
  const int K = P.grid_clusters > 1 ? P.grid_clusters : 1;
  if (!launch_shape_ok(C, K * C)) {  // uniform over the launch: every CTA returns here
    if (blockIdx.x == 0 && threadIdx.x == 0 && P.info) P.info[ASCHED_INFO_STATUS] = ASCHED_E_INVALID;
    return;
  }
  const int rank = C > 1 ? static_cast<int>(cluster_rank()) : 0;
  const int cid = K > 1 ? static_cast<int>(blockIdx.x) / C : 0;
  solve_one<PEN, DL, DEBUG, BIG, false>(P, P.lay, C, rank, K, cid);
}

}  // namespace

namespace asched_kernels {
namespace {
template <bool PEN, bool DL>
void* full_of(bool debug, bool big) {
  if (debug) return big ? reinterpret_cast<void*>(&tabu_kernel<PEN, DL, true, true>)
                        : reinterpret_cast<void*>(&tabu_kernel<PEN, DL, true, false>);
  return big ? reinterpret_cast<void*>(&tabu_kernel<PEN, DL, false, true>)
             : reinterpret_cast<void*>(&tabu_kernel<PEN, DL, false, false>);
}
}  // namespace
void* full(bool pen, bool dl, bool debug, bool big) {
  if (pen) return dl ? full_of<true, true>(debug, big) : full_of<true, false>(debug, big);
  return dl ? full_of<false, true>(debug, big) : full_of<false, false>(debug, big);
}
}  // namespace asched_kernels
