// Batches: many instances in one launch.
#include "search.cuh"
#include "kernels.h"
#include "instance.cuh"

namespace {

// Processing order: instances by decreasing neighbourhood size (ties by index), so the
// persistent CTAs start the longest solves first. Also resets the ticket counter.
__global__ void batch_order_kernel(int32_t B, const int32_t* veh_off, const int32_t* mis_off, int32_t* work) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
    const int64_t nb = moves_of(mis_off[b + 1] - mis_off[b], veh_off[b + 1] - veh_off[b]);
    int r = 0;
    for (int k = 0; k < B; ++k) {
      const int64_t nk = moves_of(mis_off[k + 1] - mis_off[k], veh_off[k + 1] - veh_off[k]);
      r += (nk > nb) || (nk == nb && k < b);
    }
    work[1 + r] = b;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) work[0] = 0;
}

// CL: the launch is made of thread-block clusters of Q.run.cluster CTAs and each instance
// is solved by a whole cluster (the same search as asched_solve with that cluster size):
// rank 0 takes the ticket and the other CTAs read it from rank 0's shared memory between
// two cluster barriers.
template <bool PEN, bool DL, bool CL>
__global__ void __launch_bounds__(kMaxThreads, 1) tabu_batch_kernel(const __grid_constant__ BParams Q) {
  __shared__ int s_ticket;
  const int C = CL ? Q.run.cluster : 1;
  if (CL && !launch_shape_ok(C, 0)) {  // uniform over the launch: nothing is solved
    if (blockIdx.x == 0)
      for (int b = threadIdx.x; b < Q.B; b += blockDim.x)
        Q.info[static_cast<int64_t>(b) * ASCHED_INFO_LEN + ASCHED_INFO_STATUS] = ASCHED_E_INVALID;
    return;
  }
  const int rank = CL ? static_cast<int>(cluster_rank()) : 0;
  while (true) {
    if (rank == 0 && threadIdx.x == 0) s_ticket = atomicAdd(&Q.work[0], 1);
    int k;
    if (CL) {
      cluster_sync_unaligned();  // thread 0 of rank 0 arrives from its claim
      k = rank == 0 ? s_ticket : ld_peer_i32(mapa_rank(smem_u32(&s_ticket), 0));
      cluster_sync_unaligned();  // every CTA has read it before rank 0 takes the next
    } else {
      __syncthreads();
      k = s_ticket;
      __syncthreads();
    }
    if (k >= Q.B) break;
    const int b = Q.work[1 + k];
    KParams P = Q.run;
    const int lo = Q.loc_off[b], vo = Q.veh_off[b], mo = Q.mis_off[b];
    P.L = Q.loc_off[b + 1] - lo;
    P.V = Q.veh_off[b + 1] - vo;
    P.M = Q.mis_off[b + 1] - mo;
    P.travel = Q.travel + Q.travel_off[b];
    P.veh_base = Q.veh_base + vo;
    P.veh_type = Q.veh_type ? Q.veh_type + vo : nullptr;
    P.pickup = Q.pickup + mo;
    P.delivery = Q.delivery + mo;
    P.heli_only = Q.heli_only ? Q.heli_only + mo : nullptr;
    P.deadline = Q.deadline ? Q.deadline + mo : nullptr;
    P.cap = Q.duty_cap[b];
    P.horizon = Q.horizon[b];
    P.out_off = Q.out_off + vo + b;
    P.out_route = Q.out_route + mo;
    P.out_flight = Q.out_flight + vo;
    P.out_over = Q.out_over + vo;
    P.info = Q.info + static_cast<int64_t>(b) * ASCHED_INFO_LEN;
    search_instance<PEN, DL>(P, C, rank, Q.compact != 0, Q.table_words, Q.limit_words);
    __syncthreads();  // the next instance's prologue reuses shared memory
  }
}

}  // namespace

namespace asched_kernels {
namespace {
template <bool PEN, bool DL>
void* batch_of(bool clusters) {
  return clusters ? reinterpret_cast<void*>(&tabu_batch_kernel<PEN, DL, true>)
                  : reinterpret_cast<void*>(&tabu_batch_kernel<PEN, DL, false>);
}
}  // namespace
void* batch(bool pen, bool dl, bool clusters) {
  if (pen) return dl ? batch_of<true, true>(clusters) : batch_of<true, false>(clusters);
  return dl ? batch_of<false, true>(clusters) : batch_of<false, false>(clusters);
}
void* batch_order() { return reinterpret_cast<void*>(&batch_order_kernel); }
}  // namespace asched_kernels
