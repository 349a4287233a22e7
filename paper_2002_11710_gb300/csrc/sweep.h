// What the sweep kernels share: their parameters and small helpers.
#pragma once

#include <stddef.h>
#include <stdint.h>

struct SwParams {
  int32_t B, nt, tenure, max_sweeps, lambda, accept_worse, repair, trace_cap;
  const int32_t* vehicle_order;  // at veh_off[b], or NULL
  const int32_t* mission_rank;   // at mis_off[b], or NULL
  const int32_t* loc_off;
  const int32_t* veh_off;
  const int32_t* mis_off;
  const int64_t* travel_off;
  const int32_t* travel;
  const int32_t* veh_base;
  const int32_t* veh_type;
  const int32_t* pickup;
  const int32_t* delivery;
  const int32_t* heli_only;
  const int32_t* deadline;
  const int32_t* duty_cap;
  const int32_t* horizon;
  int32_t* out_off;
  int32_t* out_route;
  int32_t* out_flight;
  int32_t* out_over;
  int32_t* info;
  uint32_t* trace_move;
  int32_t* trace_z;
};

namespace asched_kernels {
// One warp per instance, for instances of at most kWarpNodes missions and vehicles together.
constexpr int kWarpNodes = 64;
void* sweep_warp(bool pen, bool dl, bool tabu);
size_t sweep_warp_bytes(int M, int V, int nt, bool tabu);  // shared memory of one instance
}  // namespace asched_kernels
