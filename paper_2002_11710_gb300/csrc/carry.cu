// The single-instance search with carried move values.
#include "search.cuh"
#include "kernels.h"

namespace {

template <bool PEN, bool DL, class TT>
__global__ void __launch_bounds__(kMaxThreads, 1) carry_kernel(const __grid_constant__ KParams P) {
  const int C = P.cluster;
  if (!launch_shape_ok(C, C)) {  // uniform over the launch: every CTA returns here
    if (blockIdx.x == 0 && threadIdx.x == 0 && P.info) P.info[ASCHED_INFO_STATUS] = ASCHED_E_INVALID;
    return;
  }
  const int rank = C > 1 ? static_cast<int>(cluster_rank()) : 0;
  carry_solve<PEN, DL, TT>(P, P.lay, C, rank);
}

}  // namespace

namespace asched_kernels {
namespace {
template <bool PEN, bool DL>
void* carry_of(bool t16) {
  return t16 ? reinterpret_cast<void*>(&carry_kernel<PEN, DL, CTab16>)
             : reinterpret_cast<void*>(&carry_kernel<PEN, DL, CTab32>);
}
}  // namespace
void* carry(bool pen, bool dl, bool t16) {
  if (pen) return dl ? carry_of<true, true>(t16) : carry_of<true, false>(t16);
  return dl ? carry_of<false, true>(t16) : carry_of<false, false>(t16);
}
}  // namespace asched_kernels
