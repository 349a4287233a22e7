// Serving: a persistent launch that solves requests as the host publishes them.
#include "search.cuh"
#include "kernels.h"
#include "instance.cuh"

namespace {

__device__ __forceinline__ int ld_volatile_i32(const int32_t* p) { return *reinterpret_cast<const volatile int32_t*>(p); }

// CL: the launch is made of thread-block clusters of Q.run.cluster CTAs and each request
// is solved by a whole cluster (the same search as asched_solve with that cluster size):
// rank 0 claims the ticket and the others read it from rank 0's shared memory between
// two cluster barriers. Their wait at the barrier ends when rank 0 arrives, which its own
// bounded claim loop guarantees.
template <bool PEN, bool DL, bool CL>
__global__ void __launch_bounds__(kMaxThreads, 1) serve_kernel(const __grid_constant__ SParams Q) {
  __shared__ int s_ticket;
  const int C = CL ? Q.run.cluster : 1;
  if (CL && !launch_shape_ok(C, 0)) return;  // uniform over the launch; nothing is served
  const int rank = CL ? static_cast<int>(cluster_rank()) : 0;
  if (threadIdx.x == 0) atomicAdd(&Q.control[ASCHED_CTRL_STARTED], 1);
  uint64_t idle_since = global_ns();
  while (true) {
    if (rank == 0 && threadIdx.x == 0) {
      int got;
      while (true) {
        const int pub = ld_volatile_i32(&Q.control[ASCHED_CTRL_PUBLISHED]);
        const int cl = ld_volatile_i32(&Q.control[ASCHED_CTRL_CLAIMED]);
        if (cl < pub) {
          if (atomicCAS(&Q.control[ASCHED_CTRL_CLAIMED], cl, cl + 1) == cl) {
            got = cl;
            break;
          }
          continue;
        }
        if (ld_volatile_i32(&Q.control[ASCHED_CTRL_STOP])) {
          got = -1;
          break;
        }
        if (static_cast<int64_t>(global_ns() - idle_since) > Q.idle_ns) {
          atomicAdd(&Q.control[ASCHED_CTRL_IDLE_EXITS], 1);
          got = -1;
          break;
        }
        __nanosleep(1000);
      }
      s_ticket = got;
    }
    int t;
    if (CL) {
      cluster_sync_unaligned();  // thread 0 of rank 0 arrives from its claim loop
      t = rank == 0 ? s_ticket : ld_peer_i32(mapa_rank(smem_u32(&s_ticket), 0));
      cluster_sync_unaligned();  // every CTA has read it before rank 0 claims the next
    } else {
      __syncthreads();
      t = s_ticket;
      __syncthreads();
    }
    if (t < 0) break;
    const int slot = ld_volatile_i32(&Q.ring[t % Q.ring_len]);
    const int32_t* in = Q.slot_data + static_cast<int64_t>(slot) * Q.slot_words;
    int32_t* out = Q.slot_out + static_cast<int64_t>(slot) * Q.out_words;
    const int L = gin(in), V = gin(in + 1), M = gin(in + 2);
    KParams P = Q.run;
    P.L = L;
    P.V = V;
    P.M = M;
    P.cap = gin(in + 3);
    P.horizon = gin(in + 4);
    const int flags = gin(in + 5);
    const int32_t* vb = in + ASCHED_SLOT_HEADER + Q.nt * Q.Lc * Q.Lc;
    P.travel = in + ASCHED_SLOT_HEADER;
    P.veh_base = vb;
    P.veh_type = vb + Q.Vc;
    P.pickup = vb + 2 * Q.Vc;
    P.delivery = P.pickup + Q.Mc;
    P.heli_only = (flags & 1) ? P.delivery + Q.Mc : nullptr;
    P.deadline = (flags & 2) ? P.delivery + 2 * Q.Mc : nullptr;
    P.out_off = out;
    P.out_route = out + Q.Vc + 1;
    P.out_flight = P.out_route + Q.Mc;
    P.out_over = P.out_flight + Q.Vc;
    P.info = P.out_over + Q.Vc;
    const bool sizes_ok = L >= 1 && L <= Q.Lc && V >= 1 && V <= Q.Vc && M >= 0 && M <= Q.Mc &&
                          (DL == ((flags & 2) != 0));
    if (sizes_ok) {
      if (!search_instance<PEN, DL>(P, C, rank, Q.compact != 0, Q.table_words, Q.limit_words) && rank == 0 &&
          threadIdx.x == 0)
        P.info[ASCHED_INFO_STATUS] = ASCHED_E_TOO_LARGE;
    } else if (rank == 0 && threadIdx.x == 0) {
      P.info[ASCHED_INFO_STATUS] = ASCHED_E_INVALID;
    }
    __syncthreads();
    if (rank == 0 && threadIdx.x == 0) {
      __threadfence_system();
      *reinterpret_cast<volatile int32_t*>(&Q.done[slot]) = gin(in + 6);
      atomicAdd(&Q.control[ASCHED_CTRL_SERVED], 1);
    }
    idle_since = global_ns();
  }
}

}  // namespace

namespace asched_kernels {
namespace {
template <bool PEN, bool DL>
void* serve_of(bool clusters) {
  return clusters ? reinterpret_cast<void*>(&serve_kernel<PEN, DL, true>)
                  : reinterpret_cast<void*>(&serve_kernel<PEN, DL, false>);
}
}  // namespace
void* serve(bool pen, bool dl, bool clusters) {
  if (pen) return dl ? serve_of<true, true>(clusters) : serve_of<true, false>(clusters);
  return dl ? serve_of<false, true>(clusters) : serve_of<false, false>(clusters);
}
}  // namespace asched_kernels
