// The paper's per-mission sweeps (see sweep.cu) for small instances: one warp per instance,
// the schedule in registers.
//
// Positions 0..n-1 hold the routes one after another, vehicle 0 first, each route's missions
// followed by its end M + v; position p is lane p mod 32, register p / 32. "Insert j before
// the node at p" is then candidate p, the order (vehicle, insertion point) of equal candidates is the order
// of positions, the points of a vehicle before its first infeasible one are a mask of
// lower lanes, and a move is a shift of the positions between its two ends: no linked
// lists, atomics or barriers. A position's record (legs, limits, its vehicle's flight, its
// mission's removal) is computed again after a move only, so a trial costs two gathers of
// travel times and one reduction.
//
// Travel times between nodes (a mission's delivery or a vehicle's base to a mission's pickup
// or a base) are gathered once into shared memory, as 16-bit words, row per end node: both
// gathers of a trial are then free of bank conflicts, while a matrix per resident instance
// (22 KB each, 30 instances) did not fit L1 and a column of it took a cache line per lane.
// Times above 32,767 are read from the matrix itself (H false).
//
// A trial whose mission was tried before, with no move applied since and none of its
// stamps still standing then, gives the same answer, no move, and is only counted.
//
// Bound by the chains of dependent shared-memory loads, votes and reductions of a trial and of
// a placement, and by instruction fetch, with 20 warps on an SM. Against one CTA of 32 threads
// with linked lists and times from L1 and L2: 16,384 paper-sized instances, Algorithm 2,
// 708 -> 356 us; 5,120 runs of Algorithm 3 in random orders 387 -> 195 us. Reading and checking
// the matrices takes 72 us of the first.
#include <cuda_runtime.h>

#include "asched.h"
#include "sweep.h"

namespace {

constexpr int kIdShift = 13;
constexpr int kNone = 0x7FFFFFFF;
constexpr int kFixed = -0x7FFFFFFF - 1;  // removal record of a mission that may not leave

__device__ __forceinline__ int pos0(int x) { return x > 0 ? x : 0; }

// Shared memory of an instance of N nodes, in bytes from the start.
struct WarpLayout {
  int times, row;  // times: nt * N rows of `row` 16-bit words
  int mis, fl, bestfl, vtype, vord, tpos, vend, tend, rank, prank, order, list, tried, last, rem, sloc, eloc, best, tabu, total;
};

__host__ __device__ inline WarpLayout warp_layout(int M, int V, int nt, bool tabu) {
  WarpLayout y;
  const int N = M + V;
  // row / 2 odd: 32 consecutive rows' entries of a column lie in different banks
  y.row = (N + 1) / 2 * 2;
  if (y.row % 4 == 0) y.row += 2;
  int o = 0;
  y.mis = o;    o += 16 * M;  // {own leg as type 0, as type 1, arrive-by time, heli-only}
  y.fl = o;     o += 4 * V;
  y.bestfl = o; o += 4 * V;
  y.vtype = o;  o += 4 * V;
  y.vord = o;   o += 4 * V;
  y.tpos = o;   o += 4 * V;  // the vehicle's turn
  y.vend = o;   o += 4 * V;  // position of the route's end
  y.tend = o;   o += 4 * V;  // end of the vehicle's turn in the list of trials
  y.rank = o;   o += 4 * M;
  y.prank = o;  o += 4 * N;  // the same by position
  y.order = o;  o += 4 * M;  // Algorithm 1's
  y.list = o;   o += 4 * M;  // trials of a sweep
  y.tried = o;  o += 4 * M;  // step of the mission's last trial
  y.last = o;   o += 4 * M;  // last step at which one of its stamps stands
  y.rem = o;    o += 4 * M;  // what its leaving takes off its vehicle's flight
  y.sloc = o;   o += 4 * N;
  y.eloc = o;   o += 4 * N;
  y.best = o;   o += 4 * (N > 4 * V ? N : 4 * V);
  y.tabu = o;   o += tabu ? 4 * M * V : 0;
  y.times = o;  o += nt * N * y.row * 2;
  y.total = (o + 15) / 16 * 16;
  return y;
}

extern __shared__ __align__(16) unsigned char g_warp[];

__device__ __forceinline__ int32_t& word(int off, int i) { return reinterpret_cast<int32_t*>(g_warp + off)[i]; }

struct Inst {
  int b, L, V, M, N, nt, cap, horizon, lam;
  const int32_t* T;
  WarpLayout y;
};

// The time at offset o of the node-to-node times: end node row, start node column. From the
// matrix itself (H false) rows are kWideRow apart, so that an offset splits without a division,
// and their matrix rows lie where the times would (4,096 instances of 36 nodes, Algorithm 3: 329 us;
// with divisions 474, one CTA of 32 threads with linked lists 371).
constexpr int kWideRow = 64;
static_assert(kWideRow >= asched_kernels::kWarpNodes, "a column per node");
template <bool H>
__device__ __forceinline__ int time_at(const Inst& s, int o) {
  if (H) return reinterpret_cast<const int16_t*>(g_warp + s.y.times)[o];
  const int64_t r = word(s.y.times, o / kWideRow);  // offsets are at least 0
  return __ldg(s.T + r * s.L + word(s.y.sloc, o % kWideRow));
}

// The register of position p (any lane's) of all positions x.
__device__ __forceinline__ int at_pos(const int (&x)[2], int p) {
  const int a = __shfl_sync(0xffffffffu, x[0], p & 31), b = __shfl_sync(0xffffffffu, x[1], p & 31);
  return p < 32 ? a : b;
}
// The same for a position that is the same in every lane.
__device__ __forceinline__ int at_one(const int (&x)[2], int p) {
  return __shfl_sync(0xffffffffu, p < 32 ? x[0] : x[1], p & 31);
}
// The first position where the predicate holds.
__device__ __forceinline__ int first_pos(bool x0, bool x1) {
  const unsigned a = __ballot_sync(0xffffffffu, x0), b = __ballot_sync(0xffffffffu, x1);
  return a ? __ffs(a) - 1 : 31 + __ffs(b);
}

// Greedy start and sweeps of one instance, whose statics and times are in shared memory, and
// its outputs. Every step of it is in the code once, and the second register of a lane is a
// uniform branch rather than a second instantiation: the resident warps are all at different
// places, and a larger body ran out of instruction cache (a form that evaluated four trials
// side by side waited for instructions 3.9 of 9 cycles).
template <bool PEN, bool DL, bool TABU, bool H>
__device__ __forceinline__ void search(const SwParams& Q, const Inst& s) {
  const int lane = threadIdx.x & 31;
  const int M = s.M, V = s.V, N = s.N, cap = s.cap, lam = s.lam, row = H ? s.y.row : kWideRow;
  const bool two = N > 32;  // both registers are in use
  const int4* const mis = reinterpret_cast<const int4*>(g_warp + s.y.mis);
  // ---- positions: node | vehicle << 8, and their records
  constexpr int kEmpty = 0xFFFF;
  int pk[2], rowE[2], colB[2], leg[2], dep[2], lim[2], fl[2];
  bool plane[2];
  unsigned mask[2], mask0 = 0;  // lower positions of the same route: own register's; of position >= 32, register 0's
  int n = 0;                    // positions in use
  fl[1] = leg[1] = dep[1] = lim[1] = rowE[1] = colB[1] = 0;
  plane[1] = false;
  mask[1] = 0;

  // ---- mission order of Algorithm 1: heli-only first, then by (deadline, id)
  for (int m = lane; m < M; m += 32) {
    const int4 d = mis[m];
    int r = 0;
#pragma unroll 2
    for (int k = 0; k < M; ++k) {
      const int2 x = *reinterpret_cast<const int2*>(&word(s.y.mis, 4 * k + 2));
      r += (x.y > d.w) || (x.y == d.w && (x.x < d.z || (x.x == d.z && k < m)));
    }
    word(s.y.order, r) = m;
    word(s.y.last, m) = -1;
  }

  // ---- Algorithm 1's state, a vehicle per lane: row of the route's last node, entry of its
  // base in row 0 of its layer, leg home, departure from the last node, flight, missions
  int grow[2], gcol[2], gleg[2], gdep[2], gfl[2], gn[2];
  bool gplane[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int u = lane + 32 * c < V ? lane + 32 * c : 0;
    const int ty = word(s.y.vtype, u);
    gplane[c] = ty != 0;
    grow[c] = (ty * N + M + u) * row;
    gcol[c] = ty * N * row + M + u;
    gleg[c] = gdep[c] = gfl[c] = gn[c] = 0;
  }
  __syncwarp();

  bool greedy = true, repaired = false, go_on = true, dirty = false;
  int placed = 0, sweeps = 0, z = 0, z_init = 0, z_best = 0, best_step = -1, moves = 0;
  int step = 0, applied_at = -1;  // the last step that applied a move
  int status = ASCHED_OK;
  const int64_t trace0 = static_cast<int64_t>(s.b) * Q.trace_cap;
  while (true) {
    if (greedy) {
      // ---- Algorithm 1: append the mission where the objective grows least (ties: lowest
      // vehicle). With the repair flag, one that fits nowhere is tried again after a sweep
      // over the partial schedule.
      bool stuck = false;
      for (; placed < M; ++placed) {
        const int m = word(s.y.order, placed);
        const int4 d = mis[m];
        int ins[2], home[2], key[2];
        key[1] = kNone;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c && V <= 32) continue;
          const int a = time_at<H>(s, grow[c] + m) + (gplane[c] ? d.y : d.x);
          home[c] = time_at<H>(s, gcol[c] + m * row);
          ins[c] = a + home[c] - gleg[c];
          bool ok = lane + 32 * c < V && !(d.w && gplane[c]);
          if (DL) ok = ok && gdep[c] + a <= d.z && d.z + home[c] <= s.horizon;
          if (!PEN) ok = ok && gfl[c] + ins[c] <= cap;
          key[c] = ok ? ins[c] + (PEN ? lam * (pos0(gfl[c] + ins[c] - cap) - pos0(gfl[c] - cap)) : 0) : kNone;
        }
        const int least = __reduce_min_sync(0xffffffffu, min(key[0], key[1]));
        if (least == kNone) {
          stuck = true;
          break;
        }
        const int v = first_pos(key[0] == least, key[1] == least);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c && V <= 32) continue;
          if (lane + 32 * c == v) {
            word(s.y.list, m) = v | (gn[c] << 8);  // number gn of vehicle v
            ++gn[c];
            gfl[c] += ins[c];
            gleg[c] = home[c];
            gdep[c] = d.z;
            grow[c] = ((gplane[c] ? N : 0) + m) * row;
          }
        }
        repaired = false;
      }
      if (stuck && (repaired || !Q.repair || placed == 0)) {
        status = ASCHED_E_INFEASIBLE_INIT;
        break;
      }
      // ---- the vehicles' routes as positions
      __syncwarp();
      int before = 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c && V <= 32) continue;
        const int v = lane + 32 * c;
        int upto = v < V ? gn[c] + 1 : 0;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(0xffffffffu, upto, o);
          if (lane >= o) upto += x;
        }
        if (v < V) {
          const int end = before + upto - 1;
          word(s.y.vend, v) = end;
          word(s.y.best, end) = (M + v) | (v << 8);
          word(s.y.bestfl, v) = end - gn[c];
          word(s.y.fl, v) = gfl[c];
        }
        before += __shfl_sync(0xffffffffu, upto, 31);
      }
      __syncwarp();
      for (int k = lane; k < placed; k += 32) {
        const int m = word(s.y.order, k), x = word(s.y.list, m), v = x & 255;
        word(s.y.best, word(s.y.bestfl, v) + (x >> 8)) = m | (v << 8);
      }
      for (int m = lane; m < M; m += 32) word(s.y.tried, m) = -1;
      n = V + placed;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c) pk[c] = lane + 32 * c < n ? word(s.y.best, lane + 32 * c) : kEmpty;
      dirty = true;
      step = 0;
      applied_at = -1;
      if (stuck) {
        repaired = true;
      } else {  // complete: the first best schedule (its positions are in best)
        greedy = false;
        int part = 0;
        for (int v = lane; v < V; v += 32) {
          const int f = word(s.y.fl, v);
          part += f + lam * pos0(f - cap);
          word(s.y.bestfl, v) = f;
        }
        z = z_init = z_best = __reduce_add_sync(0xffffffffu, part);
      }
    }
    if (!greedy && !(go_on && sweeps < Q.max_sweeps)) break;

    // ---- one sweep: the vehicles' turns in order; a turn tries the vehicle's missions as its
    // route stands when the turn starts, in route order or by increasing rank
    const bool worse = Q.accept_worse && !greedy, trace = !greedy && Q.trace_cap > 0;
    const int z0 = z_best;
    bool applied = false;
    int t = 0, trials = 0, next = 0;  // trial, end of the list that holds, turn to list from
    while (true) {
      if (dirty) {
        // ---- records of the positions
        __syncwarp();
        unsigned ends[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) ends[c] = __ballot_sync(0xffffffffu, (pk[c] & 255) >= M && pk[c] != kEmpty);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c && !two) continue;
          const int p = lane + 32 * c;
          const int before = at_pos(pk, (p - 1) & 63) & 255, after = at_pos(pk, (p + 1) & 63) & 255;
          const bool on = p < n;
          const int nd = on ? pk[c] & 255 : M, vh = on ? pk[c] >> 8 : 0;
          const bool first = p == 0 || before >= M;
          const int pv = first ? M + vh : before;
          const int ty = word(s.y.vtype, vh);
          plane[c] = ty != 0;
          rowE[c] = (ty * N + pv) * row;
          colB[c] = ty * N * row + nd;
          fl[c] = word(s.y.fl, vh);
          dep[c] = DL && !first ? mis[pv].z : 0;
          lim[c] = s.horizon;
          if (nd >= M) {
            leg[c] = first ? 0 : time_at<H>(s, rowE[c] + nd);
            if (on) word(s.y.vend, vh) = p;
          } else {
            leg[c] = time_at<H>(s, rowE[c] + nd);
            const int4 d = mis[nd];
            const int own = ty != 0 ? d.y : d.x;
            if (DL) lim[c] = d.z - own;
            const bool single = first && after >= M;
            const int link = single ? 0 : time_at<H>(s, rowE[c] + after);
            const int r = leg[c] + own + time_at<H>(s, (ty * N + nd) * row + after) - link;
            bool ok = true;
            if (DL) {
              int nl = s.horizon;
              if (after < M) {
                const int4 x = mis[after];
                nl = x.z - (ty != 0 ? x.y : x.x);
              }
              ok = dep[c] + link <= nl;
            }
            if (!PEN) ok = ok && fl[c] - r <= cap;
            word(s.y.rem, nd) = ok || single ? r : kFixed;
          }
          // lower positions of the same route: above the last end below p
          const unsigned low = (1u << lane) - 1u;
          const unsigned e = ends[c] & low;
          mask[c] = e ? low & ~((2u << (31 - __clz(e))) - 1u) : low;
          if (c) mask0 = e ? 0u : ends[0] ? ~((2u << (31 - __clz(ends[0]))) - 1u) : ~0u;
        }
        __syncwarp();
        dirty = false;
      }
      if (t >= trials) {
        if (next >= V) break;
        // ---- the trials of the turns from `next` on, as the routes stand: mission | vehicle << 8
        // | end of the turn in the list << 16
        int before = 0;
#pragma unroll 1
        for (int c = 0; 32 * c < V; ++c) {
          const int u = lane + 32 * c;
          const bool on = u >= next && u < V;
          const int v = on ? word(s.y.vord, u) : 0;
          int upto = on ? word(s.y.vend, v) - (v > 0 ? word(s.y.vend, v - 1) + 1 : 0) : 0;
#pragma unroll 1
          for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += x;
          }
          if (on) word(s.y.tend, v) = before + upto;
          before += __shfl_sync(0xffffffffu, upto, 31);
        }
        if (Q.mission_rank) {
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if ((pk[c] & 255) < M) word(s.y.prank, lane + 32 * c) = word(s.y.rank, pk[c] & 255);
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c && !two) continue;
          const int p = lane + 32 * c, nd = pk[c] & 255, v = pk[c] >> 8;
          if (nd >= M || word(s.y.tpos, v) < next) continue;
          const int p1 = word(s.y.vend, v), p0 = v > 0 ? word(s.y.vend, v - 1) + 1 : 0;
          int at = p - p0;
          if (Q.mission_rank) {
            const int mine = word(s.y.prank, p);
            at = 0;
            for (int x = p0; x < p1; ++x) at += word(s.y.prank, x) < mine;
          }
          const int end = word(s.y.tend, v);
          word(s.y.list, end - (p1 - p0) + at) = nd | (v << 8) | (end << 16);
        }
        __syncwarp();
        trials = before;
        next = V;
        t = 0;
        continue;
      }
      // ---- one trial: mission j of vehicle i
      const int entry = word(s.y.list, t);
      const int j = entry & 255, i = (entry >> 8) & 255;
      const int4 dj = mis[j];
      const int rm = word(s.y.rem, j), tried = word(s.y.tried, j);
      bool known = tried > applied_at;
      if (TABU) known = known && word(s.y.last, j) < tried;
      bool apply = false;
      int least = kNone;
      int d[2], ins[2];
      d[1] = kNone;
      ins[1] = 0;
      if (!known && rm != kFixed) {
        int di = -rm;
        if (PEN) {
          const int fi = word(s.y.fl, i);
          di += lam * (pos0(fi - rm - cap) - pos0(fi - cap));
        }
        bool act[2], ok[2];
        act[1] = false;
        ok[1] = true;
        bool some = false;  // a candidate that would be applied, if no point before it stops its vehicle
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c && !two) continue;
          const int a = time_at<H>(s, rowE[c] + j) + (plane[c] ? dj.y : dj.x);
          const int bq = time_at<H>(s, colB[c] + j * row);
          ins[c] = a + bq - leg[c];
          ok[c] = true;
          if (DL) ok[c] = dep[c] + a <= dj.z && dj.z + bq <= lim[c];
          if (!PEN) ok[c] = ok[c] && fl[c] + ins[c] <= cap;
          d[c] = di + ins[c];
          if (PEN) d[c] += lam * (pos0(fl[c] + ins[c] - cap) - pos0(fl[c] - cap));
          const int vh = pk[c] >> 8;
          act[c] = lane + 32 * c < n && vh != i && !(dj.w && plane[c]);
          if (TABU) act[c] = act[c] && word(s.y.tabu, j * V + (act[c] ? vh : 0)) < step;
          some = some || (act[c] && ok[c] && (d[c] < 0 || worse));
        }
        if (__any_sync(0xffffffffu, some)) {
          const unsigned stop0 = __ballot_sync(0xffffffffu, act[0] && !ok[0]);
          const unsigned stop1 = __ballot_sync(0xffffffffu, act[1] && !ok[1]);
          if (!act[0] || !ok[0] || (stop0 & mask[0])) d[0] = kNone;
          if (!act[1] || !ok[1] || (stop1 & mask[1]) || (stop0 & mask0)) d[1] = kNone;
          least = __reduce_min_sync(0xffffffffu, min(d[0], d[1]));
          apply = least != kNone && (least < 0 || worse);
        }
      }
      __syncwarp();  // every lane has read j's words
      uint32_t move = ASCHED_NULL_MOVE;
      if (apply) {
        const int to = first_pos(d[0] == least, d[1] == least);
        const int from = first_pos((pk[0] & 255) == j, (pk[1] & 255) == j);
        const int target = at_one(pk, to), add = at_one(ins, to);
        const int k = target >> 8;
        // take the node at `from` out and put it before `to`, on vehicle k
        const bool down = from < to;
        const int dst = down ? to - 1 : to;
        int moved[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int p = lane + 32 * c;
          int src = p;
          if (down && p >= from && p < dst) src = p + 1;
          if (!down && p > dst && p <= from) src = p - 1;
          if (p == dst) src = from;
          moved[c] = at_pos(pk, src);
          if (p == dst) moved[c] = j | (k << 8);
        }
        pk[0] = moved[0];
        pk[1] = moved[1];
        if (lane == 0) {
          word(s.y.fl, i) -= rm;
          word(s.y.fl, k) += add;
          if (TABU && !greedy) {
            word(s.y.tabu, j * V + i) = step + Q.tenure;
            word(s.y.last, j) = step + Q.tenure;
          }
        }
        move = (static_cast<uint32_t>(j) << kIdShift) | static_cast<uint32_t>(target & 255);
        dirty = applied = true;
        applied_at = step;
        if (!greedy) {
          z += least;
          ++moves;
          if (z < z_best) {
            z_best = z;
            best_step = step;
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 2; ++c)
              if (lane + 32 * c < N) word(s.y.best, lane + 32 * c) = pk[c];
            for (int v = lane; v < V; v += 32) word(s.y.bestfl, v) = word(s.y.fl, v);
          }
        }
        // the rest of this turn goes on; later turns start from the new routes
        trials = entry >> 16;
        next = word(s.y.tpos, i) + 1;
      }
      if (lane == 0) {
        word(s.y.tried, j) = step;
        if (trace && step < Q.trace_cap) {
          if (Q.trace_move) Q.trace_move[trace0 + step] = move;
          if (Q.trace_z) Q.trace_z[trace0 + step] = z;
        }
      }
      ++t;
      ++step;
    }
    if (!greedy) {
      ++sweeps;
      go_on = Q.accept_worse ? z_best < z0 : applied;
      continue;
    }
    if (!applied) {
      status = ASCHED_E_INFEASIBLE_INIT;
      break;
    }
    // ---- back to Algorithm 1 with the routes of the repair sweep
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (lane + 32 * c >= n) continue;
      const int nd = pk[c] & 255, vh = pk[c] >> 8;
      const int idx = __popc(mask[c]) + (c ? __popc(mask0) : 0);
      if (nd < M) {
        word(s.y.list, nd) = vh | (idx << 8);
      } else {
        word(s.y.best, 4 * vh) = rowE[c];
        word(s.y.best, 4 * vh + 1) = leg[c];
        word(s.y.best, 4 * vh + 2) = dep[c];
        word(s.y.best, 4 * vh + 3) = idx;
      }
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int v = lane + 32 * c;
      if (v >= V) continue;
      grow[c] = word(s.y.best, 4 * v);
      gleg[c] = word(s.y.best, 4 * v + 1);
      gdep[c] = word(s.y.best, 4 * v + 2);
      gn[c] = word(s.y.best, 4 * v + 3);
      gfl[c] = word(s.y.fl, v);
    }
    __syncwarp();
  }
  __syncwarp();

  // ---- best schedule out: CSR from the kept positions, flight and overflow per vehicle
  const bool good = status == ASCHED_OK;
  if (good) {
    const int vo = Q.veh_off[s.b], mo = Q.mis_off[s.b];
    int32_t* off = Q.out_off + vo + s.b;
    for (int p = lane; p < N; p += 32) {
      const int x = word(s.y.best, p), nd = x & 255, vh = x >> 8;
      if (nd < M) {
        Q.out_route[mo + p - vh] = nd;
      } else {  // the end of vh's route: the next vehicle's first mission comes p - vh missions in
        off[vh + 1] = p - vh;
        const int f = word(s.y.bestfl, vh);
        if (Q.out_flight) Q.out_flight[vo + vh] = f;
        if (Q.out_over) Q.out_over[vo + vh] = pos0(f - cap);
      }
    }
    if (lane == 0) off[0] = 0;
  }
  if (lane == 0) {
    int32_t* info = Q.info + static_cast<int64_t>(s.b) * ASCHED_INFO_LEN;
    info[ASCHED_INFO_STATUS] = status;
    info[ASCHED_INFO_Z_BEST] = good ? z_best : 0;
    info[ASCHED_INFO_BEST_IT] = good ? best_step : 0;
    info[ASCHED_INFO_Z_INIT] = good ? z_init : 0;
    info[ASCHED_INFO_Z_FINAL] = good ? z : 0;
    info[ASCHED_INFO_ITERS] = sweeps;
    info[ASCHED_INFO_MOVES] = moves;
    info[ASCHED_INFO_STEPS] = good ? step : 0;
  }
}

template <bool PEN, bool DL, bool TABU>
__global__ void __launch_bounds__(32, 20) sweep_warp_kernel(const __grid_constant__ SwParams Q) {
  const int lane = threadIdx.x;
  Inst s;
  s.b = blockIdx.x;
  const int lo = Q.loc_off[s.b], vo = Q.veh_off[s.b], mo = Q.mis_off[s.b];
  s.L = Q.loc_off[s.b + 1] - lo;
  s.V = Q.veh_off[s.b + 1] - vo;
  s.M = Q.mis_off[s.b + 1] - mo;
  s.N = s.M + s.V;
  s.nt = Q.nt;
  s.cap = Q.duty_cap[s.b];
  s.horizon = Q.horizon[s.b];
  s.lam = PEN ? Q.lambda : 0;
  s.T = Q.travel + Q.travel_off[s.b];
  s.y = warp_layout(s.M, s.V, s.nt, TABU);
  const int L = s.L, V = s.V, M = s.M, N = s.N, nt = s.nt;

  // ---- load and validate (the same checks as the full-neighbourhood search)
  int bad = 0;
  for (int m = lane; m < M; m += 32) {
    const int pk = Q.pickup[mo + m], d = Q.delivery[mo + m];
    const int h = Q.heli_only ? Q.heli_only[mo + m] : 0;
    bad |= (pk < 0) | (pk >= L) | (d < 0) | (d >= L) | (pk == d) | (h < 0) | (h > 1);
    word(s.y.sloc, m) = pk;
    word(s.y.eloc, m) = d;
    word(s.y.mis, 4 * m + 2) = DL ? Q.deadline[mo + m] : 0;
    word(s.y.mis, 4 * m + 3) = h;
    word(s.y.rank, m) = Q.mission_rank ? Q.mission_rank[mo + m] : m;
  }
  for (int v = lane; v < V; v += 32) {
    const int bl = Q.veh_base[vo + v];
    const int ty = Q.veh_type ? Q.veh_type[vo + v] : 0;
    bad |= (bl < 0) | (bl >= L) | (ty < 0) | (ty >= nt);
    word(s.y.sloc, M + v) = bl;
    word(s.y.eloc, M + v) = bl;
    word(s.y.vtype, v) = ty;
    word(s.y.vord, v) = Q.vehicle_order ? Q.vehicle_order[vo + v] : v;
  }
  int maxT = 0;
  {  // the matrices, 16 bytes per load between an unaligned head and tail
    const int64_t n = static_cast<int64_t>(nt) * L * L;
    const int64_t head = min(static_cast<int64_t>((16u - (reinterpret_cast<uintptr_t>(s.T) & 15u)) & 15u) / 4, n);
    const int64_t n4 = (n - head) >> 2;
    int least = 0;
    auto see = [&](int t) {
      least = min(least, t);
      maxT = max(maxT, t);
    };
    for (int64_t x = lane; x < head; x += 32) see(__ldg(s.T + x));
    const int4* T4 = reinterpret_cast<const int4*>(s.T + head);
#pragma unroll 8
    for (int64_t x = lane; x < n4; x += 32) {
      const int4 t = __ldg(T4 + x);
      see(t.x);
      see(t.y);
      see(t.z);
      see(t.w);
    }
    for (int64_t x = head + 4 * n4 + lane; x < n; x += 32) see(__ldg(s.T + x));
    bad |= least < 0;
  }
  maxT = __reduce_max_sync(0xffffffffu, maxT);
  int status = __any_sync(0xffffffffu, bad) ? ASCHED_E_INVALID : ASCHED_OK;
  if (status == ASCHED_OK) {
    // 2 (2M + V + 2) maxT (1 + lambda) < 2^31 keeps every int32 sum in range.
    const double bound = 2.0 * (2.0 * M + V + 2.0) * static_cast<double>(maxT) * (1.0 + static_cast<double>(s.lam));
    if (!(bound < 2147483648.0)) status = ASCHED_E_OVERFLOW_GUARD;
  }
  if (status == ASCHED_OK && (Q.vehicle_order || Q.mission_rank)) {
    // the orders must be permutations (bestfl and list serve as counters here)
    for (int v = lane; v < V; v += 32) word(s.y.bestfl, v) = 0;
    for (int m = lane; m < M; m += 32) word(s.y.list, m) = 0;
    __syncwarp();
    int badp = 0;
    for (int v = lane; v < V; v += 32) {
      const int x = word(s.y.vord, v);
      if (x < 0 || x >= V) badp = 1;
      else atomicAdd(&word(s.y.bestfl, x), 1);
    }
    for (int m = lane; m < M; m += 32) {
      const int x = word(s.y.rank, m);
      if (x < 0 || x >= M) badp = 1;
      else atomicAdd(&word(s.y.list, x), 1);
    }
    __syncwarp();
    for (int v = lane; v < V; v += 32) badp |= word(s.y.bestfl, v) != 1;
    for (int m = lane; m < M; m += 32) badp |= word(s.y.list, m) != 1;
    if (__any_sync(0xffffffffu, badp)) status = ASCHED_E_INVALID;
  }
  __syncwarp();
  if (status != ASCHED_OK) {
    if (lane < ASCHED_INFO_LEN)
      Q.info[static_cast<int64_t>(s.b) * ASCHED_INFO_LEN + lane] = lane == ASCHED_INFO_STATUS ? status : 0;
    return;
  }

  for (int v = lane; v < V; v += 32) word(s.y.tpos, word(s.y.vord, v)) = v;

  // ---- in-mission legs per travel layer, times between nodes, tabu list
  for (int t = 0; t < 2; ++t)
    for (int m = lane; m < M; m += 32)
      word(s.y.mis, 4 * m + t) =
          t < nt ? __ldg(s.T + (static_cast<int64_t>(t) * L + word(s.y.sloc, m)) * L + word(s.y.eloc, m)) : 0;
  const bool half = maxT <= 32767;
  if (half) {
    int16_t* const X = reinterpret_cast<int16_t*>(g_warp + s.y.times);
    for (int c = lane; c < N; c += 32) {
      const int32_t* col = s.T + word(s.y.sloc, c);
      for (int t = 0; t < nt; ++t) {
        for (int e0 = 0; e0 < N; e0 += 12) {  // loads first: the compiler keeps them behind earlier stores
          int x[12];
#pragma unroll
          for (int k = 0; k < 12; ++k)
            x[k] = __ldg(col + static_cast<int64_t>(word(s.y.eloc, e0 + k < N ? e0 + k : N - 1)) * L);
#pragma unroll
          for (int k = 0; k < 12; ++k)
            if (e0 + k < N) X[(t * N + e0 + k) * s.y.row + c] = static_cast<int16_t>(x[k]);
        }
        col += static_cast<int64_t>(L) * L;
      }
    }
  }
  if (!half)  // matrix rows of the end nodes, by layer
    for (int x = lane; x < nt * N; x += 32) word(s.y.times, x) = x < N ? word(s.y.eloc, x) : L + word(s.y.eloc, x - N);
  if (TABU)
    for (int x = lane; x < M * V; x += 32) word(s.y.tabu, x) = -1;
  __syncwarp();

  if (half) search<PEN, DL, TABU, true>(Q, s);
  else search<PEN, DL, TABU, false>(Q, s);
}

}  // namespace

namespace asched_kernels {
namespace {
template <bool PEN, bool DL>
void* sweep_warp_of(bool tabu) {
  return tabu ? reinterpret_cast<void*>(&sweep_warp_kernel<PEN, DL, true>)
              : reinterpret_cast<void*>(&sweep_warp_kernel<PEN, DL, false>);
}
}  // namespace
void* sweep_warp(bool pen, bool dl, bool tabu) {
  if (pen) return dl ? sweep_warp_of<true, true>(tabu) : sweep_warp_of<true, false>(tabu);
  return dl ? sweep_warp_of<false, true>(tabu) : sweep_warp_of<false, false>(tabu);
}
size_t sweep_warp_bytes(int M, int V, int nt, bool tabu) { return static_cast<size_t>(warp_layout(M, V, nt, tabu).total); }
}  // namespace asched_kernels
