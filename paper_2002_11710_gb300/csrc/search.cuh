// search.cuh - GB300 (sm_103a) Tabu search for air-ambulance fleet scheduling: device code.
//
// Method: Tassone & Choudhury, "Algorithms for Optimizing Fleet Scheduling of Air
// Ambulances" (arXiv 2002.11710): model of Section 3 (obj_s, con1-con13), greedy
// start of Algorithm 1 (Section 4.1), Tabu search of Algorithm 3 (Section 4.3)
// widened to the whole relocate + swap neighbourhood every iteration. The readings
// of the paper that fix the move set, move ids, tabu attribute, aspiration and
// tie-break are stated in include/asched.h.
//
// Design (one instance per launch):
//   * One persistent launch runs every iteration. The grid is one thread-block
//     cluster of C CTAs (C = 1..16), or K such clusters for large neighbourhoods, one
//     CTA per SM. Each CTA holds a complete copy of the instance and of the search
//     state in shared memory and applies every move itself, so the only traffic
//     between CTAs per iteration is one 64-bit key per CTA: a relaxed DSMEM store of a
//     key tagged with the iteration inside a cluster, and a relaxed global store of the
//     cluster's key between clusters, each polled by the receivers with a bounded wait.
//   * Shared memory holds two node-by-mission gather tables built once per launch:
//       A[t][l][m] = T_t[l][p_m] + T_t[p_m][d_m]   (fly from location l to m's pickup, then m)
//       B[t][l][m] = T_t[d_m][l]                   (from m's delivery to location l)
//     with the mission index innermost and rows padded to a multiple of 32 words,
//     so that 32 lanes reading 32 consecutive missions of any row hit 32 banks; or,
//     for instances whose tables do not fit, the travel matrix itself in int16.
//   * The schedule is a doubly linked list over nodes (missions 0..M-1 and route
//     ends M..M+V-1), with per-node records (removal delta, gap leg, slot cost,
//     table row offsets, cap slack, deadline slacks) in an SoA. A node's records
//     depend only on its own links and vehicle and on static tables, so applying a move
//     rewrites the at most six relinked nodes in place (one warp, a lane per node), while
//     another warp takes the two routes' new flights.
//   * Every move (relocate (m, y) and swap (a, b)) is evaluated in O(1) from the
//     records and the tables; the per-thread, warp (redux.sync), CTA (shared
//     memory), cluster (DSMEM) and grid (L2) minimum of the key
//     ((delta ^ 2^31) << 32) | id is independent of how moves are split over threads,
//     so any launch shape gives the same trajectory.
//   * The tabu list is a V x M table of iteration stamps in shared memory.
//   * The batch and serving kernels run the same search per instance, one CTA or one
//     cluster each; their item lists take one more record per mission (a relocation's
//     source-route delta), relocations of four missions at a time and the pass over every
//     pair of missions in its short form, the swaps of route neighbours in a pass of their own.

#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "asched.h"

namespace {

constexpr uint32_t kSwapBit = 0x80000000u;
constexpr uint32_t kNullMove = 0xFFFFFFFFu;
constexpr uint64_t kNoKey = ~0ull;
constexpr int kMaxCluster = 16;
constexpr int kMaxGridClusters = 1024;  // clusters of one single-instance launch
constexpr int kMaxThreads = 512;  // per CTA; leaves 128 registers per thread
constexpr int kIdShift = 13;
constexpr uint32_t kIdMask = (1u << kIdShift) - 1u;
constexpr int kMaxMissions = 4095;
constexpr int kMaxNodes = 8192;
constexpr int kMaxVehicles = 1024;
constexpr int64_t kDefaultTimeoutNs = 1000000000ll;

// ------------------------------------------------------------------ layout ---------

// Per-node records. A node word packs the next node and the node's
// vehicle word: nv = next | vw << 13, vw = vehicle | plane << 10 | heli-only << 11.
//   R2[t] = {nv, removal delta}                       relocation, mission side
//   Y4[t] = {A row of prev(t), B row of t, leg prev(t) -> t, nv}   relocation, gap side
//   S4[t] = {nv, A row of prev(t), B row of next(t), slot cost}    swap side
//   D4[t] = {dep(prev t), arrive-by slack at t, slack at next(t), removal link ok}
//   PRV[t] previous node; FB[v] flight of vehicle v minus the duty cap;
//   RP[t]  (after FB) a relocation's delta on t's own route when t moves to another
//          route: removal delta plus lambda times the change of that route's overflow
//          (penalty mode), or whether the route stays within the cap (hard mode). Kept by
//          the batch and serving kernels where they evaluate item lists, whose length it
//          cuts, and not by the single-instance kernel, whose iterations wait on the apply step.
constexpr int kBufWordsPerNode = 15;

// Two table layouts. Small instances keep location x mission gather tables (int32):
//   A[t][l][m] = T_t[l][p_m] + T_t[p_m][d_m],  B[t][l][m] = T_t[d_m][l],
// row stride Mp words, so 32 lanes reading 32 consecutive missions hit 32 banks.
// Large instances ("big") keep the travel matrix itself in int16 (exact while every
// entry is below 2^15) with a row stride of Ls halves, Ls / 2 odd, so that random rows
// and random columns both spread over the banks; tabu stamps are int16 there too.
struct Layout {  // offsets in int32 words from the start of dynamic shared memory
  int A, B, tabu, cmat, wm, eloc, sloc, vtype, tyl, tym, st0, best, order, cnt, gend, gdep, gfl,
      glast, misc, mbar, warpkey, slots, gkey, total;
  int Mp, Np, Vp, buf, Ls;
  bool big;  // the int16 matrix, or the limits that come with it
  // carry layouts only (see carry.cuh)
  int rec, d4, prv, vr, ktab, itab, tb, list, rows, ccnt, expired, bound, ring, pkey;
  int S, Sp, VW;        // missions per CTA, row stride of the tables, words of a vehicle set
  int gm_log, ulog, ucap, kv;  // lanes per mission group (log2); least nodes (log2) and most number of column
                               // units; vehicles per lane of a scan unit
};

__host__ __device__ inline int round_up(int x, int k) { return (x + k - 1) / k * k; }

__host__ __device__ inline Layout make_layout(int M, int V, int L, int nt, bool big, bool rp) {
  Layout y = {};
  y.big = big;
  y.Mp = round_up(M > 0 ? M : 1, 32);
  y.Np = round_up(M + V, 4);
  y.Vp = round_up(V, 4);
  y.buf = kBufWordsPerNode * y.Np + y.Vp + (rp ? y.Np : 0);  // R2 Y4 S4 D4 PRV, FB, RP
  y.Ls = round_up(L, 2);
  if ((y.Ls / 2) % 2 == 0) y.Ls += 2;
  int o = 0;
  if (big) {
    y.A = o;     o += round_up(nt * L * y.Ls / 2, 4);  // int16 travel matrix
    y.B = y.A;
    y.tabu = o;  o += round_up(V * y.Mp / 2, 4);      // int16 stamps
  } else {
    y.A = o;     o += nt * L * y.Mp;
    y.B = o;     o += nt * L * y.Mp;
    y.tabu = o;  o += V * y.Mp;
  }
  y.cmat = o;    o += nt * y.Mp;
  y.wm = o;      o += y.Mp;
  y.eloc = o;    o += round_up(M + V + 3, 4);  // quads of missions read up to M + 2
  y.sloc = o;    o += round_up(M + V + 3, 4);
  y.vtype = o;   o += y.Vp;
  y.tyl = o;     o += y.Vp;
  y.tym = o;     o += y.Vp;
  y.st0 = o;     o += y.buf;
  y.best = o;    o += y.Np;
  y.order = o;   o += y.Mp;
  y.cnt = o;     o += y.Mp;
  y.gend = o;    o += y.Vp;
  y.gdep = o;    o += y.Vp;
  y.gfl = o;     o += y.Vp;
  y.glast = o;   o += y.Vp;
  y.misc = o;    o += 16;
  y.mbar = o;    o += 2;  // one mbarrier (8 bytes; o is even here)
  o = round_up(o, 4);
  y.warpkey = o; o += 2 * 32;
  y.slots = o;   o += 2 * 2 * kMaxCluster;
  y.gkey = o;    o += 2 * 2;  // the grid's key, per slot buffer (several clusters)
  y.total = o;
  return y;
}

// Layouts with carried move values (carry.cuh): the matrix itself (int32 with an odd row
// stride, or int16 as above) at the start, the records, and the tables of one CTA's slice
// of the missions.
constexpr int kMaxCarryTenure = 512;  // ring of moves; longer tenures take the full evaluation
__host__ __device__ inline Layout make_carry_layout(int M, int V, int L, int nt, bool dl, bool t16, bool half,
                                                    int ctas, int nwarps, int tenure) {
  Layout y = {};
  y.big = half;
  y.Mp = round_up(M > 0 ? M : 1, 32);
  y.Np = round_up(M + V, 4);
  y.Vp = round_up(V, 4);
  y.VW = (V + 31) / 32;
  y.S = M > 0 ? (M + ctas - 1) / ctas : 1;
  y.gm_log = 5;
  while (y.gm_log > 0 && (1 << (y.gm_log - 1)) >= y.S) --y.gm_log;
  const int subs = 32 >> y.gm_log;
  y.Sp = y.S | 1;  // odd: 32 vehicles' entries of one mission lie in different banks
  if (y.S <= 32) {
    // one block of missions: two nodes per lane group and unit, the entries over all warps
    y.ulog = 6 - y.gm_log;
    y.ucap = nwarps;
    y.kv = (V + subs * nwarps - 1) / (subs * nwarps);
    if (y.kv < 4) y.kv = 4;
  } else {
    const int nblk = (y.S + 31) / 32;
    y.ulog = 3;
    y.ucap = nblk * 2 > 16 ? nblk * 2 : 16;
    y.kv = V;
  }
  int o = 0;
  y.A = o;
  if (t16) {
    y.Ls = round_up(L, 2);
    if ((y.Ls / 2) % 2 == 0) y.Ls += 2;
    o += round_up(nt * L * y.Ls / 2, 4);
  } else {
    y.Ls = L | 1;
    const int64_t words = static_cast<int64_t>(nt) * L * y.Ls;
    if (words > 65536) {  // beyond any CTA's shared memory
      y.total = 1 << 28;
      return y;
    }
    o += round_up(static_cast<int>(words), 4);
  }
  y.rec = o;     o += 8 * y.Np;
  y.d4 = o;      o += dl ? 4 * y.Np : 0;
  const int64_t table = 2 * static_cast<int64_t>(V) * y.Sp;
  if (table > 65536) {
    y.total = 1 << 28;
    return y;
  }
  // K, over the prologue's scratch and the staging buffer of the int16 matrix
  const int scratch = 2 * y.Mp + 4 * y.Vp;
  const int least = scratch + (t16 ? 2048 : 0);
  y.ktab = o;
  y.order = o;
  y.cnt = o + y.Mp;
  y.gend = o + 2 * y.Mp;
  y.gdep = y.gend + y.Vp;
  y.gfl = y.gdep + y.Vp;
  y.glast = y.gfl + y.Vp;
  y.st0 = o + scratch;
  const int kwords = round_up(table > least ? static_cast<int>(table) : least, 4);
  y.buf = (kwords - scratch) & ~3;
  o += kwords;
  y.itab = o;    o += round_up(V * y.Sp, 4);
  y.cmat = o;    o += nt * y.Mp;
  y.wm = o;      o += y.Mp;
  y.eloc = o;    o += round_up(M + V + 1, 4);
  y.sloc = o;    o += round_up(M + V + 1, 4);
  y.vtype = o;   o += y.Vp;
  y.tyl = o;     o += y.Vp;
  y.tym = o;     o += y.Vp;
  y.prv = o;     o += y.Np;
  y.vr = o;      o += 4 * y.Vp;
  y.best = o;    o += y.Np;
  y.tb = o;      o += y.VW * y.Mp;
  y.list = o;    o += round_up(M + V, 8);  // two lists of 16-bit nodes
  y.rows = o;    o += round_up(y.S, 8) / 2;  // 16-bit missions
  y.ccnt = o;    o += 8;
  y.expired = o; o += 4;
  y.bound = o;   o += round_up(y.S, 4);
  y.ring = o;    o += round_up(2 * tenure, 4);
  y.pkey = o;    o += 64 * y.ucap;
  y.misc = o;    o += 16;
  y.mbar = o;    o += 2;
  o = round_up(o, 4);
  y.warpkey = o; o += 2 * 32;
  y.slots = o;   o += 2 * 2 * kMaxCluster;
  y.gkey = o;    o += 2 * 2;
  y.total = o;
  return y;
}

// Items of the full evaluation: relocations of two missions, swaps.
__host__ __device__ inline int64_t search_items(int64_t M, int64_t V) {
  return (M + V) * ((M + 1) / 2) + M * (M - 1) / 2;
}

// Whether carried move values are faster than the full evaluation, on one cluster. Full: its
// items. Carried, in the same unit (all times four): a fixed part per warp for the chain of
// table updates; P, the pairs of a node of the two changed routes and a mission (two routes of
// average length; with one vehicle its only one), each of which takes both sides of a swap; and
// V M, the entries that are scanned. With few vehicles P is most of the neighbourhood: that is
// where the line lies. On clusters a pair costs more, since every CTA keeps all nodes' records
// for a slice of the missions. Arrive-by times lengthen the full evaluation more. Fitted to both
// sides at 20 to 300 missions, 1 to 50 vehicles, 1 to 1,024 instances, 64 to 512 threads, 1 to 16
// CTAs; the rule's choice is on average 0.2 to 0.7 % slower than the better side. us an
// iteration, full / carried:
//   one instance, 512 threads:  200 missions on 1 vehicle 17.5 / 34.3, on 4 18.9 / 19.4, on 8
//     18.9 / 11.5; 100 on 4 6.3 / 8.6, on 8 6.4 / 5.5; 40 on 8 2.7 / 3.4
//   1,024 instances, 256 threads:  200 on 3 208 / 194, on 12 207 / 88; 100 on 4 48.5 / 68.6, on
//     8 48.6 / 48.1, on 20 50.1 / 37.3; 60 on 12 27.7 / 26.1; 40 on 8 19.7 / 24.0
//   a cluster of 8 CTAs of 256 threads:  200 on 12 5.8 / 6.3, on 20 6.0 / 5.5; 300 on 20
//     11.8 / 9.1; 100 on 20 3.2 / 3.7; of 512 threads, 5 missions a vehicle:  160 3.5 / 3.7, 190
//     4.4 / 4.0, 260 7.5 / 5.7
__host__ __device__ inline int64_t carry_cost(int64_t M, int64_t V, bool dl, int64_t ctas, int64_t nwarps) {
  const int64_t pairs = V == 1 ? (M + 1) * M : 2 * M * (M + V) / V, entries = V * M;
  if (ctas == 1) {
    const int64_t rest = pairs + entries < 40 * M ? pairs + entries : 40 * M;
    return dl ? 400 * nwarps + 5 * pairs + 2 * entries : 600 * nwarps + 6 * pairs + 4 * rest;
  }
  const int64_t f = ctas <= 4 ? 7 : 12, chain = (ctas <= 4 ? 600 : 450) * ctas * nwarps;
  return dl ? 400 * ctas * nwarps + f * pairs + 2 * entries : chain + 2 * f * pairs + 4 * entries;
}
__host__ __device__ inline bool carry_pays(int64_t M, int64_t V, bool dl, int64_t ctas, int64_t nwarps) {
  return 4 * search_items(M, V) > carry_cost(M, V, dl, ctas, nwarps);
}

// The layout of a search: carried move values where they fit limit_words (with the int32 matrix,
// or, where the limits of the int16 matrix hold anyway, the int16 one) and pay, or the full
// evaluation does not fit; else the full evaluation with the gather tables or the int16 matrix,
// whatever it takes. half: those limits hold (the caller asks for the
// compact layout, or the gather tables do not fit). rp: with RP records.
enum SearchKind { SEARCH_TABLES = 0, SEARCH_HALF, SEARCH_CARRY32, SEARCH_CARRY16 };
__host__ __device__ inline int pick_search(int M, int V, int L, int nt, bool dl, int ctas, int nwarps, int tenure,
                                           bool compact, bool half, bool rp, int limit_words, Layout* out) {
  const Layout full = make_layout(M, V, L, nt, half, rp);
  if (tenure <= kMaxCarryTenure && (carry_pays(M, V, dl, ctas, nwarps) || full.total > limit_words)) {
    if (!compact) {
      *out = make_carry_layout(M, V, L, nt, dl, false, half, ctas, nwarps, tenure);
      if (out->total <= limit_words) return SEARCH_CARRY32;
    }
    if (half) {
      *out = make_carry_layout(M, V, L, nt, dl, true, half, ctas, nwarps, tenure);
      if (out->total <= limit_words) return SEARCH_CARRY16;
    }
  }
  *out = full;
  return half ? SEARCH_HALF : SEARCH_TABLES;
}

// Whether the full evaluation of a batch or a request takes RP records, relocations of four
// missions and a pass of their own for neighbours: from 6 chunks of 32 items a warp on, where
// issue bounds it. Below, pairs without them are faster, since the records cost a barrier
// (20 missions, 256 threads, 1.7 chunks: 1.8 against 2.2 us an iteration); above, with them
// (1,024 instances of 100 missions on 2 vehicles, 40 chunks: 49 against 57 us; of 200 210
// against 248). With the line at 4, 300 paper-fleet instances take 3,385 us instead of 3,335 and a
// backlog of 128 requests 16,560 instead of 16,505.
constexpr int kQuadChunks = 6;
__host__ __device__ inline bool takes_quads(int M, int V, int ctas, int nwarps) {
  return search_items(M, V) > 32ll * kQuadChunks * ctas * nwarps;
}

// ------------------------------------------------------------------ parameters -----

struct KParams {
  const int32_t* travel;
  const int32_t* veh_base;
  const int32_t* veh_type;
  const int32_t* pickup;
  const int32_t* delivery;
  const int32_t* heli_only;
  const int32_t* deadline;
  int32_t L, nt, V, M, cap, horizon;
  int32_t tenure, iterations, lambda, cluster;
  int32_t grid_clusters;  // clusters cooperating on the instance (1: one cluster)
  int32_t gslot_stride;   // words (uint64) between the two global slot buffers
  uint64_t* gslots;       // [2][gslot_stride] keys of the clusters (grid_clusters > 1), zeroed
  int32_t test_withhold;  // the last CTA (cluster) does not publish its first key (tests the timeout)
  int64_t timeout_ns;
  Layout lay;
  const int32_t* init_off;
  const int32_t* init_route;
  const int32_t* tabu_in;
  int32_t dbg_it, dbg_zbest;
  int32_t* out_off;
  int32_t* out_route;
  int32_t* out_flight;
  int32_t* out_over;
  int32_t* info;
  uint32_t* traj_move;
  int32_t* traj_z;
  int32_t* dbg_delta;
  uint8_t* dbg_flags;
  uint32_t* dbg_id;
  unsigned long long* dbg_key;
};

// ------------------------------------------------------------------ PTX helpers ----

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// CTAs in this CTA's cluster as launched (1 without a cluster launch).
__device__ __forceinline__ uint32_t cluster_ctas() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

// The launch has the shape the parameters describe: C CTAs per cluster and `ctas` CTAs
// in all, in a one-dimensional grid. Kernels check this before any access to a peer's
// shared memory, whose address would not exist in a launch of another shape (for
// instance one replayed without its cluster attribute).
__device__ __forceinline__ bool launch_shape_ok(int C, int ctas) {
  return static_cast<int>(cluster_ctas()) == C && (ctas <= 0 || static_cast<int>(gridDim.x) == ctas) &&
         gridDim.y == 1 && gridDim.z == 1;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// The same cluster barrier without .aligned: for code where the threads of a warp may
// arrive from different paths (the warp is also synchronised first).
__device__ __forceinline__ void cluster_sync_unaligned() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ uint32_t mapa_rank(uint32_t local_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}

// Barrier 1 of the block as a producer-consumer pair: every thread but the waiting ones
// arrives without stopping.
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Store into a peer CTA's shared memory (relaxed, cluster scope).
__device__ __forceinline__ void st_peer_u64(uint32_t cluster_addr, uint64_t v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(cluster_addr), "l"(v) : "memory");
}

// Load a 32-bit word from a peer CTA's shared memory (ordered by a cluster barrier).
__device__ __forceinline__ int ld_peer_i32(uint32_t cluster_addr) {
  int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}

// Store into this CTA's shared memory for its other warps (relaxed, CTA scope).
__device__ __forceinline__ void st_own_u64(uint32_t cta_addr, uint64_t v) {
  asm volatile("st.relaxed.cta.shared::cta.u64 [%0], %1;" ::"r"(cta_addr), "l"(v) : "memory");
}

// Load from this CTA's shared memory, observing peers' relaxed stores.
__device__ __forceinline__ uint64_t ld_own_u64(uint32_t cta_addr) {
  uint64_t v;
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(cta_addr) : "memory");
  return v;
}

// ---- bulk copies global -> shared completing on an mbarrier (compact layout staging)
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// before the barrier's memory serves anything else (the next instance of a persistent
// launch may lay shared memory out differently)
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bytes from global src into this CTA's shared dst (both 16-byte aligned, bytes a multiple of 16)
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// OR of a flag into a word of another CTA's shared memory
__device__ __forceinline__ void red_or_peer(uint32_t cluster_addr, uint32_t v) {
  asm volatile("red.shared::cluster.or.b32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

// Keys between the clusters of one instance go through global memory (L2): relaxed
// stores and loads at GPU scope, each a single 64-bit word that carries its own tag.
__device__ __forceinline__ void st_relaxed_gpu_u64(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t ld_relaxed_gpu_u64(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Instance inputs are read through L2 only (ld.global.cg): a persistent launch reuses
// request slots whose new contents arrive by copy while it runs, and L1 is not kept
// coherent with those writes. These reads happen outside the iteration loop.
__device__ __forceinline__ int gin(const int32_t* p) { return __ldcg(p); }

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ------------------------------------------------------------------ keys -----------

// Bits 26-29 of every move id are zero (R ids < 2^26; S ids use bit 31 and bits
// 0-25), so keys crossing the cluster carry an iteration tag there: 8 | ((it >> 1) & 7).
// Slots start at 0 (tag 0), and consecutive uses of a slot buffer carry different tags.
constexpr uint64_t kTagMask = 0xFull << 26;
// Bit 30 is zero in every move id too. In a key broadcast to the CTAs of a cluster it
// means "the exchange between clusters gave up" (with a high word of all ones).
constexpr uint64_t kFailBit = 1ull << 30;
__device__ __forceinline__ uint64_t iter_tag(int it) {
  return static_cast<uint64_t>(8 | ((it >> 1) & 7)) << 26;
}

__device__ __forceinline__ uint64_t pack_key(int32_t d, uint32_t id) {
  return (static_cast<uint64_t>(static_cast<uint32_t>(d) ^ 0x80000000u) << 32) | id;
}
__device__ __forceinline__ int32_t key_delta(uint64_t k) {
  return static_cast<int32_t>(static_cast<uint32_t>(k >> 32) ^ 0x80000000u);
}

__device__ __forceinline__ uint64_t warp_min_key(uint64_t k) {
  const uint32_t hi = static_cast<uint32_t>(k >> 32), lo = static_cast<uint32_t>(k);
  const uint32_t mhi = __reduce_min_sync(0xffffffffu, hi);
  const uint32_t mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? lo : 0xffffffffu);
  return (static_cast<uint64_t>(mhi) << 32) | mlo;
}

__device__ __forceinline__ uint64_t min_u64(uint64_t a, uint64_t b) { return a < b ? a : b; }
__device__ __forceinline__ int32_t pos0(int32_t x) { return x > 0 ? x : 0; }

// ------------------------------------------------------------------ shared state ---

// All state lives in dynamic shared memory and is addressed as word offsets into this
// one array, so every access compiles to a shared-memory load or store.
extern __shared__ __align__(16) int32_t g_smem[];

struct Arr {  // an int32 array in shared memory
  int off;
  __device__ __forceinline__ int32_t& operator[](int i) const { return g_smem[off + i]; }
};

struct State {  // the per-node records (see the layout notes)
  int base, np, vp;
  __device__ __forceinline__ int2* r2() const { return reinterpret_cast<int2*>(g_smem + base); }
  __device__ __forceinline__ int4* y4() const { return reinterpret_cast<int4*>(g_smem + base + 2 * np); }
  __device__ __forceinline__ int4* s4() const { return reinterpret_cast<int4*>(g_smem + base + 6 * np); }
  __device__ __forceinline__ int4* d4() const { return reinterpret_cast<int4*>(g_smem + base + 10 * np); }
  __device__ __forceinline__ int32_t* prv() const { return g_smem + base + 14 * np; }
  __device__ __forceinline__ int32_t* fb() const { return g_smem + base + 15 * np; }
  __device__ __forceinline__ int32_t* rp() const { return g_smem + base + 15 * np + vp; }
  __device__ __forceinline__ int32_t& nv(int t) const { return g_smem[base + 2 * t]; }
};

struct Smem {
  Arr A, B, tabu, cmat, wm, eloc, sloc, vtype, tyl, tym, best, order, cnt, gend, gdep, gfl, glast, misc;
  int st0, buf, np, vp;
  int warpkey_off, slots_off, gkey_off;
  __device__ __forceinline__ State records() const { return State{st0, np, vp}; }  // the per-node records
  __device__ __forceinline__ uint64_t* warpkey() const {
    return reinterpret_cast<uint64_t*>(g_smem + warpkey_off);
  }
  __device__ __forceinline__ uint64_t* slots() const { return reinterpret_cast<uint64_t*>(g_smem + slots_off); }
  __device__ __forceinline__ uint64_t* gkey() const { return reinterpret_cast<uint64_t*>(g_smem + gkey_off); }
};

__device__ inline Smem carve(const Layout& y) {
  Smem s;
  s.A = Arr{y.A};
  s.B = Arr{y.B};
  s.tabu = Arr{y.tabu};
  s.cmat = Arr{y.cmat};
  s.wm = Arr{y.wm};
  s.eloc = Arr{y.eloc};
  s.sloc = Arr{y.sloc};
  s.vtype = Arr{y.vtype};
  s.tyl = Arr{y.tyl};
  s.tym = Arr{y.tym};
  s.st0 = y.st0;
  s.buf = y.buf;
  s.np = y.Np;
  s.vp = y.Vp;
  s.best = Arr{y.best};
  s.order = Arr{y.order};
  s.cnt = Arr{y.cnt};
  s.gend = Arr{y.gend};
  s.gdep = Arr{y.gdep};
  s.gfl = Arr{y.gfl};
  s.glast = Arr{y.glast};
  s.misc = Arr{y.misc};
  s.warpkey_off = y.warpkey;
  s.slots_off = y.slots;
  s.gkey_off = y.gkey;
  return s;
}

// misc slots
enum { MISC_BAD = 0, MISC_MAXT, MISC_Z0, MISC_GREEDY_FAIL, MISC_CSR_BAD, MISC_STAGE_FAIL, MISC_STOP, MISC_VA, MISC_VB };

struct Ctx {  // per-launch constants every thread keeps in registers
  int M, V, N, L, Mp, cap, horizon, lam;
  int heli;  // some mission is heli-only
};

// Table access for either layout. A row handle is (type offset + location) times the
// row unit: Mp words for the gather tables, 1 (a row index) for the int16 matrix.
template <bool BIG>
struct Tab {
  int A, B, tabu_off, cmat, eloc, sloc;
  int Mp, L, Ls;
  __device__ __forceinline__ int row(int tyl, int loc) const { return BIG ? tyl + loc : (tyl + loc) * Mp; }
  __device__ __forceinline__ int t16(int i) const { return reinterpret_cast<const int16_t*>(g_smem + A)[i]; }
  // A[row][m]: fly from the row's location to m's pickup, then m's own leg.
  __device__ __forceinline__ int a(int r, int m) const {
    if (BIG) return t16(r * Ls + g_smem[sloc + m]) + g_smem[cmat + (r >= L ? Mp : 0) + m];
    return g_smem[A + r + m];
  }
  // B[row][m]: from m's delivery to the row's location.
  __device__ __forceinline__ int b(int r, int m) const {
    if (BIG) {
      const int tyl = r >= L ? L : 0;
      return t16((tyl + g_smem[eloc + m]) * Ls + (r - tyl));
    }
    return g_smem[B + r + m];
  }
  // Entries of missions m0 and m0 + 1 (m0 even). The per-mission arrays start on 16-byte
  // boundaries (every layout offset is a multiple of 4 words), so the pair's locations
  // and legs come in single 64-bit loads.
  __device__ __forceinline__ int2 a2(int r, int m0) const {
    if (BIG) {
      const int2 s = *reinterpret_cast<const int2*>(g_smem + sloc + m0);
      const int2 cm = *reinterpret_cast<const int2*>(g_smem + cmat + (r >= L ? Mp : 0) + m0);
      const int base = r * Ls;
      return make_int2(t16(base + s.x) + cm.x, t16(base + s.y) + cm.y);
    }
    return *reinterpret_cast<const int2*>(g_smem + A + r + m0);
  }
  __device__ __forceinline__ int2 b2(int r, int m0) const {
    if (BIG) {
      const int tyl = r >= L ? L : 0;
      const int2 e = *reinterpret_cast<const int2*>(g_smem + eloc + m0);
      const int col = r - tyl;
      return make_int2(t16((tyl + e.x) * Ls + col), t16((tyl + e.y) * Ls + col));
    }
    return *reinterpret_cast<const int2*>(g_smem + B + r + m0);
  }
  // Entries of missions m0 .. m0 + 3 (m0 a multiple of 4), by 128-bit loads.
  __device__ __forceinline__ int4 a4(int r, int m0) const {
    if (BIG) {
      const int4 s = *reinterpret_cast<const int4*>(g_smem + sloc + m0);
      const int4 cm = *reinterpret_cast<const int4*>(g_smem + cmat + (r >= L ? Mp : 0) + m0);
      const int base = r * Ls;
      return make_int4(t16(base + s.x) + cm.x, t16(base + s.y) + cm.y, t16(base + s.z) + cm.z,
                       t16(base + s.w) + cm.w);
    }
    return *reinterpret_cast<const int4*>(g_smem + A + r + m0);
  }
  __device__ __forceinline__ int4 b4(int r, int m0) const {
    if (BIG) {
      const int tyl = r >= L ? L : 0;
      const int4 e = *reinterpret_cast<const int4*>(g_smem + eloc + m0);
      const int col = r - tyl;
      return make_int4(t16((tyl + e.x) * Ls + col), t16((tyl + e.y) * Ls + col), t16((tyl + e.z) * Ls + col),
                       t16((tyl + e.w) * Ls + col));
    }
    return *reinterpret_cast<const int4*>(g_smem + B + r + m0);
  }
  __device__ __forceinline__ int4 tabu4(int v, int m0) const {
    if (BIG) {
      const short4 w = *reinterpret_cast<const short4*>(reinterpret_cast<const int16_t*>(g_smem + tabu_off) +
                                                         v * Mp + m0);
      return make_int4(w.x, w.y, w.z, w.w);
    }
    return *reinterpret_cast<const int4*>(g_smem + tabu_off + v * Mp + m0);
  }
  __device__ __forceinline__ int tabu(int v, int m) const {
    if (BIG) return reinterpret_cast<const int16_t*>(g_smem + tabu_off)[v * Mp + m];
    return g_smem[tabu_off + v * Mp + m];
  }
  __device__ __forceinline__ int2 tabu2(int v, int m0) const {  // m0 even
    if (BIG) {
      const short2 w = *reinterpret_cast<const short2*>(reinterpret_cast<const int16_t*>(g_smem + tabu_off) +
                                                         v * Mp + m0);
      return make_int2(w.x, w.y);
    }
    return *reinterpret_cast<const int2*>(g_smem + tabu_off + v * Mp + m0);
  }
  __device__ __forceinline__ void set_tabu(int v, int m, int x) const {
    if (BIG) reinterpret_cast<int16_t*>(g_smem + tabu_off)[v * Mp + m] = static_cast<int16_t>(x);
    else g_smem[tabu_off + v * Mp + m] = x;
  }
};

template <bool BIG>
__device__ __forceinline__ Tab<BIG> make_tab(const Layout& y, int L) {
  Tab<BIG> t;
  t.A = y.A;
  t.B = y.B;
  t.tabu_off = y.tabu;
  t.cmat = y.cmat;
  t.eloc = y.eloc;
  t.sloc = y.sloc;
  t.Mp = y.Mp;
  t.L = L;
  t.Ls = y.Ls;
  return t;
}

constexpr int kNodeMask = 0x1FFF;  // next-node field of a node word
__device__ __forceinline__ int nv_next(int nv) { return nv & kNodeMask; }
__device__ __forceinline__ int nv_vw(int nv) { return (nv >> 13) & 0xFFF; }
__device__ __forceinline__ int nv_veh(int nv) { return (nv >> 13) & 0x3FF; }
__device__ __forceinline__ int vw_veh(int vw) { return vw & 0x3FF; }
__device__ __forceinline__ int vw_plane(int vw) { return (vw >> 10) & 1; }
// the vehicle part of `from` with the heli-only bit of `own`
__device__ __forceinline__ int vw_move(int from, int own) { return (from & 0x7FF) | (own & 0x800); }

// Write every record of node t into S from its links (nx, pv) and its vehicle word vw.
template <bool PEN, bool DL, bool BIG>
__device__ __forceinline__ void write_records(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                              int t, int nx, int pv, int vw) {
  // Every load comes before the first store: the stores go to the same shared array, so
  // the compiler could not move a load above one of them. Missions and route ends take the
  // same path: this is a chain on one warp that the others wait for.
  const int plane = vw_plane(vw);
  const int tyl = plane * c.L, tym = plane * c.Mp;
  const bool mission = t < c.M, nm = nx < c.M, pm = pv < c.M;
  const int tm = mission ? t : 0, nxm = nm ? nx : 0, pvm = pm ? pv : 0;
  const int rowA = tb.row(tyl, sm.eloc[pv]);
  const int rowB = tb.row(tyl, sm.sloc[t]);
  const int rowBn = tb.row(tyl, sm.sloc[nx]);
  const int ct = sm.cmat[tym + tm], cx = sm.cmat[tym + nxm];
  int wt = 0, wx = 0, wp = 0;
  if (DL) {
    wt = sm.wm[tm];
    wx = sm.wm[nxm];
    wp = sm.wm[pvm];
  }
  const int aT = tb.a(rowA, tm), bT = tb.b(rowBn, tm);
  const int aN = tb.a(rowA, nxm), bP = tb.b(mission ? rowBn : rowB, pvm);
  const int nv = nx | (vw << 13);
  const int home = pm ? bP : 0;  // from the previous mission to the end
  const int leg = nm ? aN - cx : home;
  const int slot = aT + bT;
  S.prv()[t] = pv;
  S.r2()[t] = make_int2(nv, mission ? leg - slot : 0);
  S.y4()[t] = make_int4(rowA, rowB, mission ? aT - ct : home, nv);
  S.s4()[t] = make_int4(nv, rowA, rowBn, slot);  // of missions
  if (DL) {
    const int dep = pm ? wp : 0, cn = nm ? cx : 0, wn = nm ? wx : c.horizon;
    S.d4()[t] = mission ? make_int4(dep, wt - ct, wn - cn, dep + leg + cn <= wn ? 1 : 0) : make_int4(dep, c.horizon, 0, 1);
  }
}

// The RP record of a mission: rem its removal delta, fm its route's flight minus the cap.
template <bool PEN>
__device__ __forceinline__ int source_part(const Ctx& c, int rem, int fm) {
  return PEN ? rem + c.lam * (pos0(fm + rem) - pos0(fm)) : (fm + rem <= 0 ? 1 : 0);
}

__device__ __forceinline__ uint8_t move_flags(bool feas, bool tabu, bool asp, bool adm) {
  return static_cast<uint8_t>((feas ? 1 : 0) | (tabu ? 2 : 0) | (asp ? 4 : 0) | (adm ? 8 : 0));
}

// Relocation R(m, y): take m out, put it immediately before node y. The inputs are
// already loaded: m's node word, removal delta and RP record, the gap record g of y, the
// table entries a = A[row of prev(y)][m], b = B[row of y][m], y's vehicle slack fy and
// the tabu stamp of (m, vehicle of y). zrel = z_best - Z, so the move aspires when
// delta < zrel (Z + delta < z_best). An admissible move's key replaces acc when smaller.
// HELI: the instance has heli-only missions (else the compatibility test is always true).
template <bool PEN, bool DL, bool DEBUG, bool RP, bool HELI>
__device__ __forceinline__ void reloc_one(const Smem& sm, const State& S, const Ctx& c, int y, int m, int nvm,
                                          int rem, int rp, const int4& g, int a, int b, int fy, int stamp, int it,
                                          int zrel, const KParams& P, uint64_t& acc) {
  const bool valid = RP ? (y != m) && (y != nv_next(nvm)) : (y != m) & (y != nv_next(nvm));
  const int vm = nv_veh(nvm), vy = nv_veh(g.w);
  const int ins = a + b - g.z;
  const int d = rem + ins;
  // Same route: one flight changes by d. Different routes: the source's flight by rem
  // (its part of the delta is m's RP record where kept), the target's by ins. Both are
  // computed and selected, so lanes never diverge.
  const bool same = vm == vy;
  int delta;
  bool feas;
  const int fm = RP ? 0 : S.fb()[vm];
  int4 dy = make_int4(0, 0, 0, 0);
  int w = 0, leave = 1;
  if (DL && !RP) {
    dy = S.d4()[y];
    w = sm.wm[m];
    leave = S.d4()[m].w;
  }
  if (RP) {
    const int grow = same ? d : ins;  // change of the target route's flight
    if (PEN) {
      delta = (same ? d : rp + ins) + c.lam * (pos0(fy + grow) - pos0(fy));
      feas = true;
    } else {
      delta = d;
      feas = (fy + grow <= 0) && (same || rp != 0);
    }
  } else if (PEN) {
    const int pen = same ? pos0(fy + d) : pos0(fm + rem) - pos0(fm) + pos0(fy + ins);
    delta = d + c.lam * (pen - pos0(fy));
    feas = true;
  } else {
    delta = d;
    feas = same ? (fy + d <= 0) : ((fm + rem <= 0) & (fy + ins <= 0));
  }
  // Few items a thread (a chain): no branches. Lists (RP, bound by issue): the first condition
  // that fails ends an item.
  const bool barred = HELI && ((nvm >> 24) & (g.w >> 23) & 1);  // heli-only m onto a plane
  if (HELI) feas = RP ? feas && !barred : feas & !barred;
  if (DL && RP) {
    dy = S.d4()[y];
    w = sm.wm[m];
    feas = feas && (dy.x + a <= w) && (w + b <= dy.y) && S.d4()[m].w;
  } else if (DL) {
    feas = feas & (dy.x + a <= w) & (w + b <= dy.y) & (leave != 0);
  }
  const bool tabu = stamp >= it;
  const bool asp = delta < zrel;
  const bool adm = RP ? valid && feas && (!tabu || asp) : valid & feas & (!tabu | asp);
  const uint32_t id = (static_cast<uint32_t>(m) << kIdShift) | static_cast<uint32_t>(y);
  if (DEBUG && valid) {
    const int64_t idx = static_cast<int64_t>(m) * (c.N - 2) + y - (y > m) - (y > nv_next(nvm));
    P.dbg_delta[idx] = delta;
    P.dbg_flags[idx] = move_flags(feas, tabu, asp, adm);
    if (P.dbg_id) P.dbg_id[idx] = id;
  }
  const uint64_t k = pack_key(delta, id);
  if (adm && k < acc) acc = k;
}

// Relocations of the mission pair (m0, m0 + 1), m0 even, before node y: every load
// serves both (64-bit loads of consecutive table and record entries).
template <bool PEN, bool DL, bool DEBUG, bool BIG, bool HELI>
__device__ __forceinline__ void eval_relocate_pair(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                                   int y, int m0, int it, int zrel, const KParams& P, uint64_t& acc) {
  const int4 rr = *reinterpret_cast<const int4*>(S.r2() + m0);  // {nv, rem} of m0 and m0 + 1
  const int4 g = S.y4()[y];  // A row, B row, leg into y, node word of y
  const int vy = nv_veh(g.w);
  const int2 a2 = tb.a2(g.x, m0);
  const int2 b2 = tb.b2(g.y, m0);
  const int2 st = tb.tabu2(vy, m0);
  const int fy = S.fb()[vy];
  reloc_one<PEN, DL, DEBUG, false, HELI>(sm, S, c, y, m0, rr.x, rr.y, 0, g, a2.x, b2.x, fy, st.x, it, zrel, P, acc);
  if (m0 + 1 < c.M)
    reloc_one<PEN, DL, DEBUG, false, HELI>(sm, S, c, y, m0 + 1, rr.z, rr.w, 0, g, a2.y, b2.y, fy, st.y, it, zrel, P, acc);
}

// Relocations of missions m0 .. m0 + 3 (m0 a multiple of 4) before node y, for the item lists
// of the batch and serving kernels: y's gap record, vehicle, flight and tabu row serve four
// moves, and the table rows, records and stamps of the four missions come in 128-bit loads.
template <bool PEN, bool DL, bool BIG, bool HELI>
__device__ __forceinline__ void eval_relocate_quad(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                                   int y, int m0, int it, int zrel, const KParams& P, uint64_t& acc) {
  const int4 r01 = *reinterpret_cast<const int4*>(S.r2() + m0);      // {nv, rem} of m0, m0 + 1
  const int4 r23 = *reinterpret_cast<const int4*>(S.r2() + m0 + 2);  // and of m0 + 2, m0 + 3
  const int4 rp = *reinterpret_cast<const int4*>(S.rp() + m0);
  const int4 g = S.y4()[y];  // A row, B row, leg into y, node word of y
  const int vy = nv_veh(g.w);
  const int4 a4 = tb.a4(g.x, m0);
  const int4 b4 = tb.b4(g.y, m0);
  const int4 st = tb.tabu4(vy, m0);
  const int fy = S.fb()[vy];
  reloc_one<PEN, DL, false, true, HELI>(sm, S, c, y, m0, r01.x, r01.y, rp.x, g, a4.x, b4.x, fy, st.x, it, zrel, P, acc);
  if (m0 + 1 < c.M)
    reloc_one<PEN, DL, false, true, HELI>(sm, S, c, y, m0 + 1, r01.z, r01.w, rp.y, g, a4.y, b4.y, fy, st.y, it, zrel, P, acc);
  if (m0 + 2 < c.M)
    reloc_one<PEN, DL, false, true, HELI>(sm, S, c, y, m0 + 2, r23.x, r23.y, rp.z, g, a4.z, b4.z, fy, st.z, it, zrel, P, acc);
  if (m0 + 3 < c.M)
    reloc_one<PEN, DL, false, true, HELI>(sm, S, c, y, m0 + 3, r23.z, r23.w, rp.w, g, a4.w, b4.w, fy, st.w, it, zrel, P, acc);
}

// Cost parts of swap S(a, b), each mission taking the other's place: t1 = fly from the
// end of a's predecessor to b's pickup plus b's own leg, t2 = from b's delivery to a's
// successor's start, t3 and t4 the same for a in b's place. When a and b are neighbours
// the predecessor or successor is the other mission itself (its delivery row is used).
struct SwapParts {
  int4 sa, sb;
  int t1, t2, t3, t4;
  bool adjA, adjB;
};

template <bool BIG>
__device__ __forceinline__ SwapParts swap_parts(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                                int a, int b) {
  SwapParts q;
  q.sa = S.s4()[a];
  q.sb = S.s4()[b];
  q.adjA = nv_next(q.sa.x) == b;  // a immediately before b
  q.adjB = nv_next(q.sb.x) == a;  // b immediately before a
  // A row of a mission's own delivery (needed only next to the other mission)
  const int rowEa = q.adjB ? tb.row(vw_plane(nv_vw(q.sa.x)) * c.L, sm.eloc[a]) : 0;
  const int rowEb = q.adjA ? tb.row(vw_plane(nv_vw(q.sb.x)) * c.L, sm.eloc[b]) : 0;
  q.t1 = tb.a(q.adjB ? rowEa : q.sa.y, b);
  q.t2 = tb.b(q.sa.z, q.adjA ? a : b);
  q.t3 = tb.a(q.adjA ? rowEb : q.sb.y, a);
  q.t4 = tb.b(q.sb.z, q.adjB ? b : a);
  return q;
}

// Swap S(a, b): the two missions exchange places. Aspiration and the key as in reloc_one.
// FAR: the pass over every pair of the batch and serving kernels, which takes the cost parts
// of two missions that are not neighbours (no delivery rows, no selects) and leaves
// neighbouring pairs out; those are the pairs (t, next t) of their neighbour pass.
// FAR = false handles any pair whole (the single-instance kernel's pass over every pair,
// and the neighbour pass).
template <bool PEN, bool DL, bool DEBUG, bool BIG, bool HELI, bool FAR>
__device__ __forceinline__ void eval_swap(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c, int a,
                                          int b, int it, int zrel, const KParams& P, uint64_t& acc) {
  SwapParts q;
  bool near = false;
  if (FAR) {
    q.sa = S.s4()[a];
    q.sb = S.s4()[b];
    near = nv_next(q.sa.x) == b || nv_next(q.sb.x) == a;
    q.adjA = q.adjB = false;
    q.t1 = tb.a(q.sa.y, b);
    q.t2 = tb.b(q.sa.z, b);
    q.t3 = tb.a(q.sb.y, a);
    q.t4 = tb.b(q.sb.z, a);
  } else {
    q = swap_parts<BIG>(sm, tb, S, c, a, b);
  }
  const int nva = q.sa.x, nvb = q.sb.x;
  const int va = nv_veh(nva), vb = nv_veh(nvb);
  const int da = q.t1 + q.t2 - q.sa.w;
  const int db = q.t3 + q.t4 - q.sb.w;
  const int fa = S.fb()[va], fb = S.fb()[vb];
  const bool same = va == vb;
  const int d = da + db;
  int delta;
  bool feas;
  if (PEN) {
    const int pen = same ? pos0(fa + d) - pos0(fa) : pos0(fa + da) - pos0(fa) + pos0(fb + db) - pos0(fb);
    delta = d + c.lam * pen;
    feas = true;
  } else {
    delta = d;
    feas = same ? (fa + d <= 0) : FAR ? (fa + da <= 0) && (fb + db <= 0) : ((fa + da <= 0) & (fb + db <= 0));
  }
  const bool asp = delta < zrel;
  bool tabu, adm;  // with and without branches as in reloc_one
  const bool barred = HELI && ((((nva >> 24) & (nvb >> 23)) | ((nvb >> 24) & (nva >> 23))) & 1);
  if (FAR) {
    if (HELI) feas = feas && !barred;
    if (DL) {
      const int4 xa = S.d4()[a], xb = S.d4()[b];
      const int wa = sm.wm[a], wb = sm.wm[b];
      feas = feas && xa.x + q.t1 <= wb && wb + q.t2 <= xa.z && xb.x + q.t3 <= wa && wa + q.t4 <= xb.z;
    }
    tabu = tb.tabu(vb, a) >= it || tb.tabu(va, b) >= it;
    adm = !near && feas && (!tabu || asp);
  } else {
    if (HELI) feas = feas & !barred;
    if (DL) {
      const int4 xa = S.d4()[a], xb = S.d4()[b];
      const int wa = sm.wm[a], wb = sm.wm[b];
      const bool l1 = (q.adjB ? wa : xa.x) + q.t1 <= wb;
      const bool l2 = q.adjA | (wb + q.t2 <= xa.z);
      const bool l3 = (q.adjA ? wb : xb.x) + q.t3 <= wa;
      const bool l4 = q.adjB | (wa + q.t4 <= xb.z);
      feas = feas & l1 & l2 & l3 & l4;
    }
    tabu = (tb.tabu(vb, a) >= it) | (tb.tabu(va, b) >= it);
    adm = feas & (!tabu | asp);
  }
  const int m1 = a < b ? a : b, m2 = a < b ? b : a;
  const uint32_t id = kSwapBit | (static_cast<uint32_t>(m1) << kIdShift) | static_cast<uint32_t>(m2);
  if (DEBUG) {
    const int64_t rtot = static_cast<int64_t>(c.M) * (c.N - 2);
    const int64_t idx = rtot + static_cast<int64_t>(m1) * (2 * c.M - m1 - 1) / 2 + (m2 - m1 - 1);
    P.dbg_delta[idx] = delta;
    P.dbg_flags[idx] = move_flags(feas, tabu, asp, adm);
    if (P.dbg_id) P.dbg_id[idx] = id;
  }
  const uint64_t k = pack_key(delta, id);
  if (adm && k < acc) acc = k;
}

// One thread's share of the evaluation (see the main loop for the item list and how its
// coordinates advance); returns the least admissible key among its moves.
struct ItemCursor {
  int r_y, r_h, s_j, s_row, s_a;  // first relocation item (y, h) and swap item (j, row, a)
  int Gq, Gr, Sq, Sr, G, H, Sn;   // grid stride in both coordinate systems, list sizes
  int n_k;                        // first item of the neighbour pass (mission t)
};

template <bool PEN, bool DL, bool DEBUG, bool BIG, bool RP, bool HELI>
__device__ __forceinline__ uint64_t eval_items(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                               const ItemCursor& q, int it, int zrel, const KParams& P) {
  uint64_t key = kNoKey;
  for (int y = q.r_y, h = q.r_h; y < c.N;) {
    if (RP) eval_relocate_quad<PEN, DL, BIG, HELI>(sm, tb, S, c, y, 4 * h, it, zrel, P, key);
    else eval_relocate_pair<PEN, DL, DEBUG, BIG, HELI>(sm, tb, S, c, y, 2 * h, it, zrel, P, key);
    h += q.Gr;
    y += q.Gq;
    if (h >= q.H) {
      h -= q.H;
      ++y;
    }
  }
  for (int j = q.s_j, row = q.s_row, a = q.s_a; j < q.Sn; j += q.G) {
    int b = a + row + 1;
    if (b >= c.M) b -= c.M;
    eval_swap<PEN, DL, DEBUG, BIG, HELI, RP>(sm, tb, S, c, a, b, it, zrel, P, key);
    a += q.Sr;
    row += q.Sq;
    if (a >= c.M) {
      a -= c.M;
      ++row;
    }
  }
  // Swaps of neighbours, t and its successor (the batch and serving kernels only, which
  // are bound by instruction issue: the pass above then takes the short form of every
  // pair; the single-instance kernel, bound by the latency of its slowest warp, keeps one
  // pass over the pairs with the neighbour case inside).
  if (RP) {
    for (int t = q.n_k; t < c.M; t += q.G) {
      const int u = nv_next(S.nv(t));
      if (u < c.M) eval_swap<PEN, DL, DEBUG, BIG, HELI, false>(sm, tb, S, c, t, u, it, zrel, P, key);
    }
  }
  return key;
}

// Searches of few items per thread: a thread's relocations (m before y) and its sides of swaps
// are the same in every iteration, so their coordinates stay in registers. Each swap is shared
// by two neighbouring lanes: a lane takes its own mission's place (m, with y put there) and
// they add up by shuffles. An iteration of such a search is the chain of a few items, so its
// length counts, not the work: pairs of relocations and whole swaps, a lane each, took 1,364
// cycles of the paper fleet's iteration (24 missions), most of the warps idle.
constexpr int kNarrowItems = 2;  // per thread at most
struct NarrowItem {
  int kind;  // 0: none, 1: relocation, 2: swap, 3: relocations of m and m + 1 (the same for a warp)
  bool live;
  int m, y;
  __device__ __forceinline__ uint32_t pack() const {
    return static_cast<uint32_t>(kind) << 28 | (live ? 1u << 27 : 0u) | static_cast<uint32_t>(m) << 13 | static_cast<uint32_t>(y);
  }
  static __device__ __forceinline__ NarrowItem of(uint32_t w) {
    return NarrowItem{static_cast<int>(w >> 28), (w >> 27 & 1u) != 0, static_cast<int>(w >> 13 & 0xFFFu),
                      static_cast<int>(w & 0x1FFFu)};
  }
};

// Chunks of 32 items: relocations (singly or of two missions), then sides of swaps.
__host__ __device__ __forceinline__ int64_t narrow_chunks(int64_t M, int64_t V, bool pairs) {
  return ((M + V) * (pairs ? (M + 1) / 2 : M) + 31) / 32 + (M * (M - 1) + 31) / 32;
}

__device__ __forceinline__ NarrowItem narrow_item(int M, int N, bool pairs, int chunk) {
  const int lane = threadIdx.x & 31;
  const int H = pairs ? (M + 1) / 2 : M;  // items per node
  const int R = (N * H + 31) / 32, W = (M * (M - 1) + 31) / 32;
  NarrowItem n = {0, false, 0, 0};
  if (chunk < R) {
    const int i = 32 * chunk + lane;
    n.kind = pairs ? 3 : 1;
    n.live = i < N * H;
    n.y = n.live ? i / H : 0;
    n.m = n.live ? (i - n.y * H) << (pairs ? 1 : 0) : 0;
  } else if (chunk < R + W) {
    const int h = 32 * (chunk - R) + lane;
    n.kind = 2;
    n.live = h < M * (M - 1);
    if (n.live) {  // the pairs (a, a + row + 1 mod M), as in the main loop's swap items
      const int j = h >> 1, row = j / M, a = j - row * M;
      const int b = a + row + 1 >= M ? a + row + 1 - M : a + row + 1;
      n.m = h & 1 ? b : a;
      n.y = h & 1 ? a : b;
    }
  }
  return n;
}

template <bool PEN, bool DL, bool BIG>
__device__ __forceinline__ uint64_t eval_narrow(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                                const NarrowItem& n, int it, int zrel, const KParams& P) {
  const int m = n.m, y = n.y;
  if (n.kind == 1) {
    const int2 r = S.r2()[m];
    const int4 g = S.y4()[y];
    const int vy = nv_veh(g.w);
    const int a = tb.a(g.x, m), b = tb.b(g.y, m), stamp = tb.tabu(vy, m), fy = S.fb()[vy];
    uint64_t key = kNoKey;
    reloc_one<PEN, DL, false, false, true>(sm, S, c, y, m, r.x, r.y, 0, g, a, b, fy, stamp, it, zrel, P, key);
    return n.live ? key : kNoKey;
  }
  if (n.kind == 3) {
    uint64_t key = kNoKey;
    eval_relocate_pair<PEN, DL, false, BIG, true>(sm, tb, S, c, y, m, it, zrel, P, key);
    return n.live ? key : kNoKey;
  }
  const int4 s = S.s4()[m];
  const int nvo = S.nv(y);
  const int vm = nv_veh(s.x), vo = nv_veh(nvo);
  const bool before = nv_next(s.x) == y, after = nv_next(nvo) == m;  // m flies just before y, just after it
  const int own = tb.row(vw_plane(nv_vw(s.x)) * c.L, sm.eloc[m]);
  const int t1 = tb.a(after ? own : s.y, y), t2 = tb.b(s.z, before ? m : y);
  const int f = S.fb()[vm];
  const bool tabu = tb.tabu(vo, m) >= it;
  int4 x = make_int4(0, 0, 0, 0);
  int wm = 0, wo = 0;
  if (DL) {
    x = S.d4()[m];
    wm = sm.wm[m];
    wo = sm.wm[y];
  }
  const int mine = t1 + t2 - s.w, other = __shfl_xor_sync(0xffffffffu, mine, 1);
  const int d = mine + other;
  const bool same = vm == vo;
  int delta = d;
  bool ok = !((s.x >> 24) & (nvo >> 23) & 1);  // heli-only m onto a plane
  if (PEN) {
    const int p0 = pos0(f);
    const int pen = pos0(f + mine) - p0;
    const int both = pen + __shfl_xor_sync(0xffffffffu, pen, 1);
    delta = d + c.lam * (same ? pos0(f + d) - p0 : both);
  } else {
    ok = ok & (f + (same ? d : mine) <= 0);
  }
  if (DL) ok = ok & ((after ? wm : x.x) + t1 <= wo) & (before | (wo + t2 <= x.z));
  const unsigned pair = 3u << (threadIdx.x & 30);
  const bool feas = !(__ballot_sync(0xffffffffu, !ok) & pair);
  const bool barred = (__ballot_sync(0xffffffffu, tabu) & pair) != 0;
  const int m1 = m < y ? m : y, m2 = m < y ? y : m;
  const uint64_t k = pack_key(delta, kSwapBit | (static_cast<uint32_t>(m1) << kIdShift) | static_cast<uint32_t>(m2));
  return n.live & feas & (!barred | (delta < zrel)) ? k : kNoKey;
}

// Flight after move `id` of the source route (src) or of the target route (!src): the
// route's flight from FB plus the move's change of it, from the same records and table
// entries the evaluators use. A move inside one route changes it by the whole delta.
template <bool BIG>
__device__ __forceinline__ int moved_flight(const Smem& sm, const Tab<BIG>& tb, const State& S, const Ctx& c,
                                            uint32_t id, bool src) {
  if (!(id & kSwapBit)) {
    const int m = static_cast<int>(id >> kIdShift), y = static_cast<int>(id & kIdMask);
    const int2 r = S.r2()[m];
    const int4 g = S.y4()[y];
    const int va = nv_veh(r.x), vb = nv_veh(g.w);
    const int ins = tb.a(g.x, m) + tb.b(g.y, m) - g.z;
    const int f = S.fb()[src ? va : vb] + c.cap;
    if (va == vb) return f + r.y + ins;
    return src ? f + r.y : f + ins;
  }
  const int a = static_cast<int>((id >> kIdShift) & kIdMask), b = static_cast<int>(id & kIdMask);
  const SwapParts q = swap_parts<BIG>(sm, tb, S, c, a, b);
  const int va = nv_veh(q.sa.x), vb = nv_veh(q.sb.x);
  const int da = q.t1 + q.t2 - q.sa.w;
  const int db = q.t3 + q.t4 - q.sb.w;
  const int f = S.fb()[src ? va : vb] + c.cap;
  if (va == vb) return f + da + db;
  return src ? f + da : f + db;
}

// Links and vehicle word of node t after a move of n1 and n2 (relocation: n1 before node n2;
// swap: n1 and n2 exchange places). p1, x1 and p2, x2: the previous and next nodes of n1 and
// n2, vwa and vwb their vehicle words, all before the move; nx, pv and vw: t's own, updated.
__device__ __forceinline__ void relink(bool is_swap, int n1, int n2, int p1, int x1, int p2, int x2, int vwa, int vwb,
                                       int t, int& nx, int& pv, int& vw) {
  if (!is_swap) {  // e -> m -> s ... x -> y  becomes  e -> s ... x -> m -> y
    if (t == p1) nx = x1;
    if (t == x1) pv = p1;
    if (t == p2) nx = n1;
    if (t == n2) pv = n1;
    if (t == n1) {
      nx = n2;
      pv = p2;
      vw = vw_move(vwb, vw);
    }
  } else if (x1 == n2) {  // pa -> a -> b -> nb  becomes  pa -> b -> a -> nb
    if (t == p1) nx = n2;
    if (t == x2) pv = n1;
    if (t == n2) {
      pv = p1;
      nx = n1;
    }
    if (t == n1) {
      pv = n2;
      nx = x2;
    }
  } else if (x2 == n1) {  // pb -> b -> a -> na  becomes  pb -> a -> b -> na
    if (t == p2) nx = n1;
    if (t == x1) pv = n2;
    if (t == n1) {
      pv = p2;
      nx = n2;
    }
    if (t == n2) {
      pv = n1;
      nx = x1;
    }
  } else {
    if (t == p1) nx = n2;
    if (t == x1) pv = n2;
    if (t == p2) nx = n1;
    if (t == x2) pv = n1;
    if (t == n1) {
      pv = p2;
      nx = x2;
      vw = vw_move(vwb, vwa);
    }
    if (t == n2) {
      pv = p1;
      nx = x1;
      vw = vw_move(vwa, vwb);
    }
  }
}

// ------------------------------------------------------------------ the kernel -----

// The compact layout's int16 matrix, row t*L + r of layer t at T16 + (t*L + r) * Ls, zero
// padded, built from the int32 input through a staging buffer: the record buffer, which
// nothing uses before the prologue writes the records. When the input is 16-byte aligned
// its words go by bulk copies completing on an mbarrier, in chunks the size of the
// buffer; every CTA copies every chunk into its own shared memory (the cluster reads the
// matrix from L2 C times; 230 KB per CTA once per solve). A block barrier after each
// chunk keeps the buffer free until every thread has converted it. Every wait is bounded
// by P.timeout_ns. With C > 1 CTAs the outcome is made the same in every CTA: a CTA whose
// copy gave up ORs a flag into rank 0's shared memory, and every CTA reads it after a
// cluster barrier. Entries are checked (>= 0) and their maximum taken on the way.
// Returns true on a timeout (in every CTA of the cluster when one timed out).
__device__ __forceinline__ bool stage_matrix16(const KParams& P, const Layout& lay, int C, int& bad, int& maxT) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int L = P.L, nt = P.nt, Ls = lay.Ls, pad = lay.Ls - P.L;
  int16_t* T16 = reinterpret_cast<int16_t*>(g_smem + lay.A);
  for (int i = tid; i < nt * L * pad; i += nthr) {
    const int r = i / pad;
    T16[r * Ls + L + (i - r * pad)] = 0;
  }
  auto put = [&](int g, int x) {
    bad |= x < 0;
    maxT = x > maxT ? x : maxT;
    const int r = g / L;
    T16[r * Ls + (g - r * L)] = static_cast<int16_t>(x);
  };
  const int words = nt * L * L;
  const bool aligned = (reinterpret_cast<uintptr_t>(P.travel) & 15u) == 0;
  const int bulk = aligned ? (words & ~3) : 0;  // words that go by bulk copies (16-byte units)
  for (int g = bulk + tid; g < words; g += nthr) put(g, gin(P.travel + g));
  const uint32_t fail_addr = smem_u32(&g_smem[lay.misc + MISC_STAGE_FAIL]);
  // Every CTA has zeroed its misc words (prologue 1) before any peer may OR into them.
  if (C > 1) cluster_sync_unaligned();
  bool gave_up = false;  // this CTA's wait ran out
  uint32_t phase = 0;
  if (bulk > 0) {
    int32_t* stage = g_smem + lay.st0;
    const int cap = lay.buf & ~3;
    const uint32_t bar = smem_u32(g_smem + lay.mbar);
    if (tid == 0) {
      mbar_init(bar, 1);
      mbar_fence_init();
    }
    __syncthreads();
    for (int c0 = 0; c0 < bulk; c0 += cap, phase ^= 1u) {
      const int n = bulk - c0 < cap ? bulk - c0 : cap;
      if (tid == 0) {
        // the block's reads of the previous chunk come before the copy overwrites it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(bar, static_cast<uint32_t>(n) * 4u);
        bulk_g2s(smem_u32(stage), P.travel + c0, static_cast<uint32_t>(n) * 4u, bar);
      }
      bool ok = mbar_try_wait(bar, phase);
      if (!ok) {
        const uint64_t t0 = global_ns();
        while (!(ok = mbar_try_wait(bar, phase))) {
          if (static_cast<int64_t>(global_ns() - t0) > P.timeout_ns) break;
        }
      }
      if (!__syncthreads_and(ok)) {
        gave_up = true;
        break;
      }
      for (int i = tid; i < n; i += nthr) put(c0 + i, stage[i]);
      __syncthreads();
    }
    if (gave_up) {  // let the copy still in flight land (bounded) before the buffer is reused
      const uint64_t t0 = global_ns();
      while (!mbar_try_wait(bar, phase) && static_cast<int64_t>(global_ns() - t0) < P.timeout_ns) {
      }
    }
    __syncthreads();  // nobody waits on the barrier after this
    if (tid == 0) mbar_inval(bar);
  }
  if (C == 1) return gave_up;
  if (gave_up && tid == 0) red_or_peer(mapa_rank(fail_addr, 0), 1u);
  cluster_sync_unaligned();
  const bool stop = ld_peer_i32(mapa_rank(fail_addr, 0)) != 0;
  cluster_sync_unaligned();  // nobody reads rank 0's flag after this
  return stop;
}

// Prologue 1 of a search: static per-mission and per-node data, range-checked (this
// thread's share; the flag says whether an entry was out of range). The caller zeroes the
// misc words first and synchronises afterwards. nodes: entries of the location arrays.
__device__ __forceinline__ int load_statics(const KParams& P, const Smem& sm, int Mp, int nodes, int& any_heli) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int M = P.M, V = P.V, N = P.M + P.V, L = P.L, nt = P.nt;
  int bad = 0;
  for (int i = tid; i < Mp; i += nthr) {
    if (i < M) {
      const int p = gin(P.pickup + i), d = gin(P.delivery + i);
      const int h = P.heli_only ? gin(P.heli_only + i) : 0;
      bad |= (p < 0) | (p >= L) | (d < 0) | (d >= L) | (p == d) | (h < 0) | (h > 1);
      any_heli |= h != 0;
      sm.wm[i] = P.deadline ? gin(P.deadline + i) : 0;
      sm.eloc[i] = d;
      sm.sloc[i] = p;
      sm.cnt[i] = 0;
    } else {
      sm.wm[i] = 0;
    }
  }
  for (int v = tid; v < V; v += nthr) {
    const int b = gin(P.veh_base + v);
    const int ty = P.veh_type ? gin(P.veh_type + v) : 0;
    bad |= (b < 0) | (b >= L) | (ty < 0) | (ty >= nt);
    sm.eloc[M + v] = b;
    sm.sloc[M + v] = b;
    sm.vtype[v] = ty;
    sm.tyl[v] = ty * L;
    sm.tym[v] = ty * Mp;
  }
  for (int i = N + tid; i < nodes; i += nthr) {  // padding read by pairs or quads of missions
    sm.eloc[i] = 0;
    sm.sloc[i] = 0;
  }
  return bad;
}

// Prologue 3 of a search: the initial schedule as links in S0 (the caller's CSR, or
// Algorithm 1 on the device). Every thread of the block calls it and gets the same status.
template <bool PEN, bool DL, class TAB, class LINKS>
__device__ __forceinline__ int initial_schedule(const KParams& P, const Smem& sm, const TAB& tb, const LINKS& S0,
                                                const Ctx& c) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int M = c.M, V = c.V;
  int status = ASCHED_OK;
  if (P.init_off) {
    int csr_bad = 0;
    for (int v = tid; v < V; v += nthr) {
      const int o0 = gin(P.init_off + v), o1 = gin(P.init_off + v + 1);
      if (o0 < 0 || o1 < o0 || o1 > M || (v == 0 && o0 != 0) || (v == V - 1 && o1 != M)) {
        csr_bad = 1;
        continue;
      }
      int prev = M + v;
      const int vw = nv_vw(S0.nv(M + v));
      for (int k = o0; k < o1; ++k) {
        const int m = gin(P.init_route + k);
        if (m < 0 || m >= M) {
          csr_bad = 1;
          break;
        }
        atomicAdd(&sm.cnt[m], 1);
        S0.nv(prev) = (S0.nv(prev) & ~kNodeMask) | m;
        S0.prv()[m] = prev;
        S0.nv(m) = (vw | ((P.heli_only ? gin(P.heli_only + m) : 0) << 11)) << 13;
        prev = m;
      }
      S0.nv(prev) = (S0.nv(prev) & ~kNodeMask) | (M + v);
      S0.prv()[M + v] = prev;
    }
    csr_bad = __syncthreads_or(csr_bad);
    if (!csr_bad) {
      int dup = 0;
      for (int m = tid; m < M; m += nthr) dup |= sm.cnt[m] != 1;
      csr_bad = __syncthreads_or(dup);
    }
    if (csr_bad) status = ASCHED_E_INVALID;
  } else {
    // Mission order: heli-only first, then by deadline, then by id.
    for (int m = tid; m < M; m += nthr) {
      const int hm = (P.heli_only && gin(P.heli_only + m)) ? 0 : 1, wmv = DL ? sm.wm[m] : 0;
      int r = 0;
      for (int k = 0; k < M; ++k) {
        const int hk = (P.heli_only && gin(P.heli_only + k)) ? 0 : 1, wk = DL ? sm.wm[k] : 0;
        r += (hk < hm) || (hk == hm && (wk < wmv || (wk == wmv && k < m)));
      }
      sm.order[r] = m;
    }
    __syncthreads();
    if (warp == 0) {
      for (int v = lane; v < V; v += 32) {
        sm.glast[v] = M + v;
        sm.gend[v] = sm.eloc[M + v];
        sm.gdep[v] = 0;
        sm.gfl[v] = 0;
      }
      __syncwarp();
      int fail = 0;
      for (int k = 0; k < M && !fail; ++k) {
        const int m = sm.order[k];
        const int w = sm.wm[m];
        const int heli = P.heli_only ? gin(P.heli_only + m) : 0;
        uint64_t best = kNoKey;
        for (int v = lane; v < V; v += 32) {
          const int tyl = sm.tyl[v];
          const int bl = sm.eloc[M + v];
          const int a = tb.a(tb.row(tyl, sm.gend[v]), m);
          const int bret = tb.b(tb.row(tyl, bl), m);
          const int last = sm.glast[v];
          const int old = last == M + v ? 0 : tb.b(tb.row(tyl, bl), last);
          const int app = a + bret - old;
          const int f = sm.gfl[v];
          bool ok = !(heli && sm.vtype[v] != 0);
          if (DL) ok = ok && (sm.gdep[v] + a <= w) && (w + bret <= c.horizon);
          int score;
          if (PEN) {
            score = app + c.lam * (pos0(f + app - c.cap) - pos0(f - c.cap));
          } else {
            ok = ok && (f + app <= c.cap);
            score = app;
          }
          if (ok) best = min_u64(best, pack_key(score, static_cast<uint32_t>(v)));
        }
        best = warp_min_key(best);
        if (best == kNoKey) {
          fail = 1;
          break;
        }
        if (lane == 0) {
          const int v = static_cast<int>(static_cast<uint32_t>(best));
          const int tyl = sm.tyl[v];
          const int bl = sm.eloc[M + v];
          const int last = sm.glast[v];
          const int a = tb.a(tb.row(tyl, sm.gend[v]), m);
          const int bret = tb.b(tb.row(tyl, bl), m);
          const int old = last == M + v ? 0 : tb.b(tb.row(tyl, bl), last);
          S0.nv(last) = (S0.nv(last) & ~kNodeMask) | m;
          S0.prv()[m] = last;
          S0.nv(m) = (M + v) | ((nv_vw(S0.nv(M + v)) | (heli << 11)) << 13);
          S0.prv()[M + v] = m;
          sm.glast[v] = m;
          sm.gend[v] = sm.eloc[m];
          sm.gdep[v] = w;
          sm.gfl[v] += a + bret - old;
        }
        __syncwarp();
      }
      if (lane == 0) sm.misc[MISC_GREEDY_FAIL] = fail;
    }
    __syncthreads();
    if (sm.misc[MISC_GREEDY_FAIL]) status = ASCHED_E_INFEASIBLE_INIT;
  }
  return status;
}

// Prologue 4 of a search: route flights (left in sm.gfl), every node's records through
// write(t, next, prev, vehicle word, flight), the schedule's feasibility (returned) and its
// objective (left in MISC_Z0; the caller synchronises before reading it).
template <bool PEN, bool DL, class TAB, class LINKS, class WRITE>
__device__ __forceinline__ bool start_records(const Smem& sm, const TAB& tb, const LINKS& S0, const Ctx& c,
                                              WRITE&& write) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int M = c.M, V = c.V, N = c.N, L = c.L;
  const Arr fl0 = sm.gfl;  // flight sums (greedy scratch is free now)
  __syncthreads();
  for (int v = tid; v < V; v += nthr) fl0[v] = 0;
  __syncthreads();
  for (int t = tid; t < N; t += nthr) {
    const int pv = S0.prv()[t];
    const int vw = nv_vw(S0.nv(t));
    const int tyl = vw_plane(vw) * L;
    int contrib;
    if (t < M) contrib = tb.a(tb.row(tyl, sm.eloc[pv]), t);
    else contrib = pv == t ? 0 : tb.b(tb.row(tyl, sm.sloc[t]), pv);
    atomicAdd(&fl0[vw_veh(vw)], contrib);
  }
  __syncthreads();
  int infeasible = 0;
  for (int t = tid; t < N; t += nthr) {
    const int nv = S0.nv(t), pv = S0.prv()[t];
    const int vw = nv_vw(nv);
    const int f = fl0[vw_veh(vw)];
    const int tyl = vw_plane(vw) * L;
    write(t, nv_next(nv), pv, vw, f);
    if (t < M) {
      infeasible |= (vw >> 11) & (vw >> 10) & 1;
      if (DL) {
        const int dep = pv < M ? sm.wm[pv] : 0;
        infeasible |= dep + tb.a(tb.row(tyl, sm.eloc[pv]), t) > sm.wm[t];
      }
    } else {
      if (!PEN) infeasible |= f > c.cap;
      if (DL && pv != t) infeasible |= sm.wm[pv] + tb.b(tb.row(tyl, sm.sloc[t]), pv) > c.horizon;
    }
  }
  const bool stop = __syncthreads_or(infeasible);
  if (warp == 0) {
    int z = 0;
    for (int v = lane; v < V; v += 32) {
      const int f = fl0[v];
      z += f + (PEN ? c.lam * pos0(f - c.cap) : 0);
    }
    z = __reduce_add_sync(0xffffffffu, z);
    if (lane == 0) sm.misc[MISC_Z0] = z;
  }
  return !stop;
}

// The least of the CTAs' keys of iteration `it`, from each CTA's own (gk, the same in all
// its threads): inside the cluster by DSMEM, between K clusters through L2. Every wait is
// bounded; timed_out is set when one ran out. Every thread of the block calls it.
__device__ __forceinline__ uint64_t exchange_keys(const KParams& P, const Smem& sm, int C, int rank, int K, int cid,
                                                  int it, uint64_t gk, bool& timed_out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (C > 1) {
    // Push this CTA's key, tagged with the iteration, into slot [it & 1][rank] of
    // every CTA; then every warp polls its own C slots until all carry this
    // iteration's tag (bounded by the timeout).
    const int sb = it & 1;
    const uint64_t tag = iter_tag(it);
    const bool withhold = P.test_withhold && K == 1 && it == 0 && rank == C - 1;  // test hook
    if (warp == 0 && lane < C && !withhold) {
      const uint32_t slot_addr = smem_u32(&sm.slots()[sb * kMaxCluster + rank]);
      st_peer_u64(mapa_rank(slot_addr, lane), (gk & ~kTagMask) | tag);
    }
    const uint32_t my_slot = smem_u32(&sm.slots()[sb * kMaxCluster + (lane < C ? lane : 0)]);
    uint64_t v = ld_own_u64(my_slot);
    bool ok = __all_sync(0xffffffffu, (v & kTagMask) == tag);
    if (!ok) {
      const uint64_t t0 = global_ns();
      while (true) {
        v = ld_own_u64(my_slot);
        ok = __all_sync(0xffffffffu, (v & kTagMask) == tag);
        if (ok) break;
        // warp-uniform decision: lane 0's clock decides for the warp
        const bool late = __shfl_sync(0xffffffffu, (int64_t)(global_ns() - t0) > P.timeout_ns, 0);
        if (late) break;
      }
    }
    if (!ok) {
      timed_out = true;
    } else {
      gk = warp_min_key(lane < C ? v : kNoKey) & ~kTagMask;
      if ((gk >> 32) == 0xFFFFFFFFull) gk = kNoKey;  // real deltas never reach 2^31 - 1
    }
  }
  if (K > 1) {
    // Between clusters: rank 0 of each cluster stores the cluster's key, tagged, into
    // global slot [it & 1][cid]; warp 0 of every CTA polls the K slots until all carry
    // this iteration's tag (bounded), takes the least and stores it, tagged, into its
    // own CTA's shared memory, where every warp polls it. A wait that gives up is
    // stored as a key with kFailBit. (Every CTA polling L2 itself measured faster than
    // rank 0 polling and pushing the key to its peers over DSMEM; more polling warps
    // per CTA, or every CTA publishing its own key, slower.) The slots were zeroed
    // before the launch; a slot buffer is reused two iterations later, when every CTA
    // has read it (a cluster publishes for it + 1 only after its CTAs have read all
    // keys of it, the cluster exchange of it + 1 coming first).
    const int sb = it & 1;
    const uint64_t tag = iter_tag(it);
    const uint32_t gk_addr = smem_u32(&sm.gkey()[sb]);
    if (warp == 0) {
      uint64_t* gs = P.gslots + static_cast<int64_t>(sb) * P.gslot_stride;
      const bool withhold = P.test_withhold && it == 0 && cid == K - 1;  // test hook
      if (rank == 0 && lane == 0 && !timed_out && !withhold)
        st_relaxed_gpu_u64(gs + cid, (gk & ~(kTagMask | kFailBit)) | tag);
      bool ok = !timed_out;
      uint64_t m = kNoKey;
      if (ok) {
        const uint64_t t0 = global_ns();
        while (true) {
          bool mine = true;
          uint64_t mk = kNoKey;
          for (int k = lane; k < K; k += 32) {
            const uint64_t v = ld_relaxed_gpu_u64(gs + k);
            mine = mine && (v & kTagMask) == tag;
            mk = min_u64(mk, v);
          }
          if (__all_sync(0xffffffffu, mine)) {
            m = warp_min_key(mk);
            break;
          }
          if (__shfl_sync(0xffffffffu, static_cast<int64_t>(global_ns() - t0) > P.timeout_ns, 0)) {
            ok = false;
            break;
          }
        }
      }
      const uint64_t msg = ok ? ((m & ~kTagMask) | tag) : ((0xFFFFFFFFull << 32) | kFailBit | tag);
      if (lane == 0) st_own_u64(gk_addr, msg);
    }
    if (!timed_out) {
      uint64_t v = ld_own_u64(gk_addr);
      bool got = __all_sync(0xffffffffu, (v & kTagMask) == tag);
      if (!got) {
        const uint64_t t0 = global_ns();
        while (true) {
          v = ld_own_u64(gk_addr);
          got = __all_sync(0xffffffffu, (v & kTagMask) == tag);
          if (got) break;
          if (__shfl_sync(0xffffffffu, static_cast<int64_t>(global_ns() - t0) > P.timeout_ns, 0)) break;
        }
      }
      if (!got || (v & kFailBit)) {
        timed_out = true;
      } else {
        gk = v & ~kTagMask;
        if ((gk >> 32) == 0xFFFFFFFFull) gk = kNoKey;
      }
    }
  }
  return gk;
}

// Whether a key names nodes of this instance (or no move).
__device__ __forceinline__ bool key_names_nodes(uint64_t gk, int M, int N) {
  if (gk == kNoKey) return true;
  const uint32_t id = static_cast<uint32_t>(gk);
  if (id & kSwapBit) {
    const uint32_t a = (id >> kIdShift) & kIdMask, b = id & kIdMask;
    return a < b && b < static_cast<uint32_t>(M);
  }
  const uint32_t m = id >> kIdShift, y = id & kIdMask;
  return m < static_cast<uint32_t>(M) && y < static_cast<uint32_t>(N) && y != m;
}

// Epilogue of a search: the best schedule (links in sm.best) in CSR form, flights and
// overflows, by the whole block of the lead CTA. Returns the status.
__device__ __forceinline__ int write_schedule(const KParams& P, const Smem& sm, const Ctx& c) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int M = c.M, V = c.V, L = c.L;
  const Arr lens = sm.gfl;  // scratch reuse (V entries)
  int walk_bad = 0;
  for (int v = tid; v < V; v += nthr) {
    int n = 0, t = sm.best[M + v];
    while (t != M + v && n <= M) {
      if (t < 0 || t >= M) {
        walk_bad = 1;
        break;
      }
      ++n;
      t = sm.best[t];
    }
    lens[v] = n;
    walk_bad |= n > M;
  }
  walk_bad = __syncthreads_or(walk_bad);
  if (tid == 0 && !walk_bad) {
    int o = 0;
    for (int v = 0; v < V; ++v) {
      P.out_off[v] = o;
      o += lens[v];
    }
    P.out_off[V] = o;
    walk_bad = o != M;
    sm.misc[MISC_CSR_BAD] = walk_bad;
  }
  __syncthreads();
  if (sm.misc[MISC_CSR_BAD]) walk_bad = 1;
  if (!walk_bad) {
    for (int v = tid; v < V; v += nthr) {
      const int32_t* T = P.travel + static_cast<int64_t>(sm.vtype[v]) * L * L;
      const int bl = sm.eloc[M + v];
      int o = 0;
      for (int w = 0; w < v; ++w) o += lens[w];
      int f = 0, prevloc = bl, t = sm.best[M + v];
      while (t != M + v) {
        P.out_route[o++] = t;
        f += gin(T + prevloc * L + sm.sloc[t]) + gin(T + sm.sloc[t] * L + sm.eloc[t]);
        prevloc = sm.eloc[t];
        t = sm.best[t];
      }
      if (lens[v] > 0) f += gin(T + prevloc * L + bl);
      if (P.out_flight) P.out_flight[v] = f;
      if (P.out_over) P.out_over[v] = pos0(f - c.cap);
    }
  } else {
    return ASCHED_E_INVALID;
  }
  return ASCHED_OK;
}

__device__ __forceinline__ void write_info(int32_t* info, int status, int zbest, int best_it, int z0, int z, int it) {
  info[ASCHED_INFO_STATUS] = status;
  info[ASCHED_INFO_Z_BEST] = zbest;
  info[ASCHED_INFO_BEST_IT] = best_it;
  info[ASCHED_INFO_Z_INIT] = z0;
  info[ASCHED_INFO_Z_FINAL] = z;
  info[ASCHED_INFO_ITERS] = it;
  info[6] = 0;
  info[7] = 0;
}

// One complete search (prologue, every iteration, epilogue) of the instance in P by
// the K clusters of C CTAs each (this CTA is `rank` in cluster `cid`), with shared
// memory laid out by lay. Every CTA holds the whole state and applies every move; CTA 0
// of cluster 0 writes the outputs.
template <bool PEN, bool DL, bool DEBUG, bool BIG, bool RP>
__device__ __forceinline__ void solve_one(const KParams& P, const Layout& lay, const int C, const int rank,
                                          const int K, const int cid) {
  const bool lead = rank == 0 && cid == 0;
  const Smem sm = carve(lay);
  const Tab<BIG> tb = make_tab<BIG>(lay, P.L);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  Ctx c;
  c.M = P.M;
  c.V = P.V;
  c.N = P.M + P.V;
  c.L = P.L;
  c.Mp = lay.Mp;
  c.cap = P.cap;
  c.horizon = P.horizon;
  c.lam = P.lambda;
  const int M = c.M, V = c.V, N = c.N, L = c.L, Mp = c.Mp, nt = P.nt;
  int status = ASCHED_OK;

  // ---- prologue 1: static per-mission / per-node data and validation
  if (tid < 16) sm.misc[tid] = 0;
  __syncthreads();
  int any_heli = 0;
  int bad = load_statics(P, sm, Mp, round_up(N + 3, 4), any_heli);
  int maxT = 0;
  if (!BIG) {  // the compact layout checks the matrix while it stages it (prologue 2)
    for (int i = tid; i < nt * L * L; i += nthr) {
      const int x = gin(P.travel + i);
      bad |= x < 0;
      maxT = x > maxT ? x : maxT;
    }
  }
  if (__syncthreads_or(bad)) status = ASCHED_E_INVALID;
  c.heli = __syncthreads_or(any_heli);
  if (BIG && status == ASCHED_OK) {
    // ---- prologue 1b: the int16 matrix, staged through shared memory by bulk copies,
    // checked as it is converted
    int tbad = 0;
    const bool timed_out = stage_matrix16(P, lay, C, tbad, maxT);
    if (__syncthreads_or(tbad)) status = ASCHED_E_INVALID;
    if (timed_out) status = ASCHED_E_TIMEOUT;  // the same in every CTA of the cluster
  }
  maxT = __reduce_max_sync(0xffffffffu, maxT);
  if (lane == 0) atomicMax(&sm.misc[MISC_MAXT], maxT);
  __syncthreads();
  if (BIG && status == ASCHED_OK && sm.misc[MISC_MAXT] > 32767) status = ASCHED_E_TOO_LARGE;
  if (status == ASCHED_OK) {
    // 2 (2M + V + 2) maxT (1 + lambda) < 2^31 keeps every int32 sum in range.
    const double bound = 2.0 * (2.0 * M + V + 2.0) * static_cast<double>(sm.misc[MISC_MAXT]) *
                         (1.0 + (PEN ? static_cast<double>(c.lam) : 0.0));
    if (!(bound < 2147483648.0)) status = ASCHED_E_OVERFLOW_GUARD;
  }

  // ---- prologue 2: gather tables, in-mission legs, tabu stamps, route ends
  const State S0 = sm.records();
  if (status == ASCHED_OK) {
    if (!BIG) {
      for (int i = tid; i < nt * L * Mp; i += nthr) {
        const int r = i / Mp, m = i - r * Mp;
        const int t = r / L, l = r - t * L;
        int av = 0, bv = 0;
        if (m < M) {
          const int32_t* T = P.travel + static_cast<int64_t>(t) * L * L;
          const int p = sm.sloc[m], d = sm.eloc[m];
          av = gin(T + l * L + p) + gin(T + p * L + d);
          bv = gin(T + d * L + l);
        }
        sm.A[i] = av;
        sm.B[i] = bv;
      }
    }
    for (int i = tid; i < nt * Mp; i += nthr) {
      const int t = i / Mp, m = i - t * Mp;
      int cv = 0;
      if (m < M) {
        const int32_t* T = P.travel + static_cast<int64_t>(t) * L * L;
        cv = gin(T + sm.sloc[m] * L + sm.eloc[m]);
      }
      sm.cmat[i] = cv;
    }
    for (int i = tid; i < V * Mp; i += nthr) {
      const int v = i / Mp, m = i - v * Mp;
      tb.set_tabu(v, m, (P.tabu_in && m < M) ? gin(P.tabu_in + static_cast<int64_t>(m) * V + v) : -1);
    }
    for (int v = tid; v < V; v += nthr) {
      S0.nv(M + v) = (M + v) | ((v | ((sm.vtype[v] != 0 ? 1 : 0) << 10)) << 13);
      S0.prv()[M + v] = M + v;
    }
  }
  __syncthreads();

  // ---- prologue 3: initial schedule (caller's CSR, or Algorithm 1 on the device)
  if (status == ASCHED_OK) status = initial_schedule<PEN, DL>(P, sm, tb, S0, c);

  // ---- prologue 4: flights, records, initial objective and feasibility
  int Z = 0;
  if (status == ASCHED_OK) {
    const bool ok = start_records<PEN, DL>(sm, tb, S0, c, [&](int t, int nx, int pv, int vw, int f) {
      write_records<PEN, DL, BIG>(sm, tb, S0, c, t, nx, pv, vw);
      if (t >= M) S0.fb()[t - M] = f - c.cap;
      else if (RP) S0.rp()[t] = source_part<PEN>(c, S0.r2()[t].y, f - c.cap);
    });
    if (!ok) status = ASCHED_E_INFEASIBLE_INIT;
    for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S0.nv(t));
    for (int i = tid; i < 2 * kMaxCluster; i += nthr) sm.slots()[i] = 0;
    if (tid < 2) sm.gkey()[tid] = 0;
    __syncthreads();
    Z = sm.misc[MISC_Z0];
  }

  // ---- main loop
  int zbest = Z, best_it = -1, it = 0;
  const bool looped = status == ASCHED_OK;  // uniform over the cluster
  if (looped) {
    if (C > 1) cluster_sync_all();
    // Static assignment over the item list [relocation pairs (N * ceil(M/2)) | swaps
    // (M(M-1)/2) | neighbour swaps (M, with RP records only)]: chunks of 32 consecutive items
    // go round-robin to (CTA, warp) over the K * C CTAs of the grid, so every CTA gets an
    // equal share and the lanes of a warp take consecutive items. A relocation item i is
    // (y, h) = divmod(i, H) for missions 2h and 2h + 1 (with RP records for missions 4h ..
    // 4h + 3); a swap item j is (row, a) = divmod(j, M) with b = (a + row + 1) mod M, which
    // lists every pair a != b once (with RP records neighbours in a route are left out there,
    // and a neighbour item t swaps mission t with its successor when that is a mission).
    // Coordinates advance by G without dividing.
    const int CT = K * C;
    const int G = CT * nthr;
    const int g = lane + 32 * (cid * C + rank + CT * warp);
    const int H = RP ? (M + 3) / 4 : (M + 1) / 2;  // relocation items per node y
    const int Rn = N * H;
    const int Sn = M * (M - 1) / 2;
    int r_y = N, r_h = 0, s_j = Sn, s_row = 0, s_a = 0, Gq = 0, Gr = 0, Sq = 0, Sr = 0, n_k = M;
    if (M > 0) {
      Gq = G / H;
      Gr = G - Gq * H;
      Sq = G / M;
      Sr = G - Sq * M;
      if (g < Rn) {
        r_y = g / H;
        r_h = g - r_y * H;
      }
      const int k = g < Rn ? (Rn - g + G - 1) / G : 0;  // relocation items of this thread
      s_j = g + k * G - Rn;
      if (s_j < Sn) {
        s_row = s_j / M;
        s_a = s_j - s_row * M;
      }
      const int k2 = g < Rn + Sn ? (Rn + Sn - g + G - 1) / G : 0;  // items before the neighbour pass
      n_k = g + k2 * G - (Rn + Sn);
    }
    const ItemCursor cursor{r_y, r_h, s_j, s_row, s_a, Gq, Gr, Sq, Sr, G, H, Sn, n_k};
    // One item a thread, with relocations singly if they fit, else two missions an item; or two.
    // Measured on single searches, narrow against the general lists: 10 missions (6 warps,
    // pairs) 291 -> 209 us for 200 iterations; 24 missions of the paper's fleet (64 warps, one
    // round) 1,734 -> 1,074 us for 1,000; 61 missions (192 warps, pairs) 1,754 -> 1,589 us with
    // the copies. Up to four rounds lost: 100 missions (3.6 rounds) 8.7 ms against 7.7 ms.
    const int64_t threads32 = static_cast<int64_t>(CT) * nwarps;
    const int64_t single = narrow_chunks(M, V, false), paired = narrow_chunks(M, V, true);
    const bool narrow = !DEBUG && !RP && (single <= kNarrowItems * threads32);
    const bool pairs = single > threads32 && paired <= threads32;
    uint32_t item[kNarrowItems];
#pragma unroll
    for (int k = 0; k < kNarrowItems; ++k)
      item[k] = narrow ? narrow_item(M, N, pairs, cid * C + rank + CT * (warp + nwarps * k)).pack() : 0u;
    const int iters = DEBUG ? 1 : P.iterations;
    bool copy_best = false;  // the last move improved the best schedule
    for (it = 0; it < iters; ++it) {
      const State S = S0;
      const int it_eval = DEBUG ? P.dbg_it : it;
      const int zb_eval = DEBUG ? P.dbg_zbest : zbest;
      // z_best - Z, clamped to int32 (a caller's z_best is arbitrary in DEBUG mode; every
      // delta lies well inside the int32 range, so the clamp changes no comparison)
      const int64_t zr = static_cast<int64_t>(zb_eval) - Z;
      const int zrel = static_cast<int>(zr < INT32_MIN ? INT32_MIN : (zr > INT32_MAX ? INT32_MAX : zr));
      uint64_t key = kNoKey;
      if (narrow) {
        // one after another through the same code: unrolled, the copies outgrow the instruction cache
        uint32_t i0 = item[0], i1 = item[1];
        static_assert(kNarrowItems == 2, "the items above");
#pragma unroll 1
        while (i0 != 0u) {
          key = min_u64(key, eval_narrow<PEN, DL, BIG>(sm, tb, S, c, NarrowItem::of(i0), it, zrel, P));
          i0 = i1;
          i1 = 0u;
        }
      } else {
        key = c.heli ? eval_items<PEN, DL, DEBUG, BIG, RP, true>(sm, tb, S, c, cursor, it_eval, zrel, P)
                     : eval_items<PEN, DL, DEBUG, BIG, RP, false>(sm, tb, S, c, cursor, it_eval, zrel, P);
      }
      if (copy_best) {
        for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S.nv(t));
      }
      key = warp_min_key(key);
      if (lane == 0) sm.warpkey()[warp] = key;
      __syncthreads();
      uint64_t gk = warp_min_key(lane < nwarps ? sm.warpkey()[lane] : kNoKey);
      bool timed_out = false;
      gk = exchange_keys(P, sm, C, rank, K, cid, it, gk, timed_out);
      // A chosen move must name nodes of this instance; anything else ends the solve
      // (gk is the same in every thread of the grid, so this decision is too).
      const bool bad_key = !timed_out && !key_names_nodes(gk, M, N);
      copy_best = false;
      if (DEBUG) {
        if (lead && tid == 0 && !timed_out) *P.dbg_key = gk;
      } else {
        // ---- apply the chosen move, in place: a node's records depend only on its own links
        // and vehicle and on static tables, so at most six nodes change. One warp rewrites
        // them, a node per lane, another takes the routes' new flights, a third (if there is
        // one) the stamps and the trajectory; the others go straight to the last barrier,
        // where all wait for the longest of these chains. (Every warp rewriting the changed
        // routes' nodes it owns, between two barriers, took 1,214 cycles of an iteration on
        // the paper-shaped instance; with flights and stamps on one warp and the trajectory
        // on the nodes' 870.)
        const bool moved = !timed_out && !bad_key && gk != kNoKey;
        const uint32_t id = static_cast<uint32_t>(gk);
        const bool is_swap = (id & kSwapBit) != 0;
        // the move's nodes (relocation: m = n1 before y = n2; swap: a = n1, b = n2); node 0
        // without a move, so that the loads below need not wait for that to be known
        const int n1 = moved ? static_cast<int>((id >> kIdShift) & kIdMask) : 0, n2 = moved ? static_cast<int>(id & kIdMask) : 0;
        if (moved) {
          Z += key_delta(gk);
          if (Z < zbest) {
            zbest = Z;
            best_it = it;
            copy_best = true;
          }
        }
        const int wstamp = nwarps > 2 ? 2 : 1;
        const int readers = nwarps > 2 ? 96 : 64;  // threads that read the move's records before warp 0 writes
        if (warp == 0) {
          const int nv1 = S.nv(n1), nv2 = S.nv(n2);
          const int p1 = S.prv()[n1], p2 = S.prv()[n2];
          const int x1 = nv_next(nv1), x2 = nv_next(nv2);
          int t = n1;
          if (lane == 1) t = n2;
          if (lane == 2) t = p1;
          if (lane == 3) t = x1;
          if (lane == 4) t = p2;
          if (lane == 5) t = x2;
          const int nvt = S.nv(t);
          int nx = nv_next(nvt), pv = S.prv()[t], vw = nv_vw(nvt);
          relink(is_swap, n1, n2, p1, x1, p2, x2, nv_vw(nv1), nv_vw(nv2), t, nx, pv, vw);
          named_sync(1, readers);
          if (moved && lane < 6) write_records<PEN, DL, BIG>(sm, tb, S, c, t, nx, pv, vw);
        } else if (warp <= wstamp) {
          const int va = nv_veh(S.nv(n1)), vb = nv_veh(S.nv(n2));
          if (warp == 1) {
            if (RP && lane == 0) {
              sm.misc[MISC_VA] = moved ? va : -1;
              sm.misc[MISC_VB] = moved ? vb : -1;
            }
            const int f = moved ? moved_flight<BIG>(sm, tb, S, c, id, lane == 0) : 0;
            named_arrive(1, readers);
            if (moved && (lane == 0 || (lane == 1 && va != vb))) S.fb()[lane == 0 ? va : vb] = f - c.cap;
          } else {
            named_arrive(1, readers);
          }
          if (warp == wstamp) {
            if (moved && (lane == 0 || (lane == 1 && is_swap)))
              tb.set_tabu(lane == 0 ? va : vb, lane == 0 ? n1 : n2, it + P.tenure);
            if (lead && lane == 2 && !timed_out) {
              if (P.traj_move) P.traj_move[it] = gk == kNoKey ? kNullMove : id;
              if (P.traj_z) P.traj_z[it] = Z;
            }
          }
        }
      }
      const bool gone = timed_out || bad_key;  // a warp's own: one may time out alone
      bool stop = gone;
      if (K * C > 1) stop = __syncthreads_or(gone);
      else __syncthreads();
      if (stop) {
        if (gone) sm.misc[MISC_STOP] = bad_key ? ASCHED_E_INVALID : ASCHED_E_TIMEOUT;
        __syncthreads();
        status = sm.misc[MISC_STOP];
        break;
      }
      if (RP) {  // the RP records of the changed routes, from their new flights
        const int va = sm.misc[MISC_VA], vb = sm.misc[MISC_VB];
        for (int t = tid; t < M; t += nthr) {
          const int2 r = S0.r2()[t];
          const int v = nv_veh(r.x);
          if (v == va || v == vb) S0.rp()[t] = source_part<PEN>(c, r.y, S0.fb()[v]);
        }
        __syncthreads();
      }
    }
    if (copy_best) {
      for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S0.nv(t));
    }
    __syncthreads();
  }

  // ---- epilogue: best schedule in CSR form (the lead CTA writes every output)
  if (lead && !DEBUG && status == ASCHED_OK && P.out_off) status = write_schedule(P, sm, c);
  if (lead && tid == 0 && P.info) write_info(P.info, status, zbest, best_it, sm.misc[MISC_Z0], Z, it);
  // No CTA may leave while a peer can still write into its shared memory.
  if (C > 1 && looped) cluster_sync_unaligned();
}

#include "carry.cuh"

}  // namespace
