// Parameters of the batch and serving kernels, and the kernels by their template options: the
// boundary between the translation units of the device code and the host side (asched.cu).
#pragma once

#include "search.cuh"

namespace {

__host__ __device__ inline int64_t moves_of(int64_t M, int64_t V) { return M * (M + V - 2) + M * (M - 1) / 2; }

// ------------------------------------------------------------------ batches --------

// Many instances in one launch. Instance b's arrays start at its offsets in the
// concatenated inputs; outputs are concatenated the same way. work[0] is a queue
// ticket counter (zeroed by batch_order_kernel), work[1 + k] the k-th instance to
// solve (largest first).
struct BParams {
  KParams run;  // tenure, iterations, lambda, nt, timeout; no instance pointers
  int32_t B;
  int32_t table_words;  // gather tables up to this size do without the int16 limits
  int32_t limit_words;  // shared memory of a CTA by which the form of a search is chosen (see pick_search)
  int32_t compact;      // always take the int16 matrix
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
  int32_t* work;
};

// ------------------------------------------------------------------ serving --------

// A persistent launch that serves requests as the host publishes them. Each request
// sits in a fixed-capacity slot (inputs) with a matching output slot; the host writes
// a slot, appends its index to the ring and raises control[PUBLISHED], all by copies
// ordered on one stream. A CTA takes the next ticket, solves that slot's instance with
// the same per-instance search as asched_solve, and writes the request's sequence
// number to done[slot]. Every wait is bounded: the launch ends when control[STOP] is
// set and every published ticket is taken, or after idle_ns without a new ticket.
struct SParams {
  KParams run;
  int32_t n_slots, ring_len, Lc, Vc, Mc, nt;
  int32_t slot_words, out_words, compact;
  int32_t limit_words;  // dynamic shared memory of the launch
  int32_t table_words;  // gather tables up to this size do without the int16 limits
  int64_t idle_ns;
  const int32_t* slot_data;
  int32_t* slot_out;
  const int32_t* ring;
  int32_t* control;
  int32_t* done;
};

__host__ __device__ inline int serve_slot_words(int Lc, int Vc, int Mc, int nt) {
  return round_up(ASCHED_SLOT_HEADER + nt * Lc * Lc + 2 * Vc + 4 * Mc, 4);
}
__host__ __device__ inline int serve_out_words(int Vc, int Mc) {
  return round_up(3 * Vc + 1 + Mc + ASCHED_INFO_LEN, 4);
}

}  // namespace

namespace asched_kernels {
void* full(bool pen, bool dl, bool debug, bool big);  // tabu_kernel: the full evaluation
void* carry(bool pen, bool dl, bool t16);             // carry_kernel: carried move values
void* batch(bool pen, bool dl, bool clusters);        // tabu_batch_kernel
void* batch_order();                                  // batch_order_kernel
void* serve(bool pen, bool dl, bool clusters);        // serve_kernel
}  // namespace asched_kernels
