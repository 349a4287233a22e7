// The Tabu search with move values carried from one iteration to the next.
//
// A move changes one or two routes (vehicles va, vb). The value of every move that touches
// neither route stays what it was, so each iteration evaluates only the columns of va and
// vb and takes the rest from two tables in shared memory, one entry per (vehicle v,
// mission m) pair:
//   I[v][m]  the least (detour, y) over the gaps y of v's route: the change of v's flight
//            when m is put before node y. It depends on v's sequence alone: the objective's
//            change is strictly increasing in the detour, and the duty cap and the tabu
//            stamp of (m, v) are the same for every y. Gaps that m's arrive-by time forbids
//            are left out.
//   K[v][m]  the least key (delta, move id) over the moves of m into v and the swaps of m
//            with a mission y of v that is not tabu on v(m).
// When a route changes, its column is computed again, and the entries of its missions in
// the other columns (their rows) are refreshed from I: a pair {m, y} can be read from
// (v(y), m) and from (v(m), y), and the column of the route that changed last holds it, so a
// row's entry keeps the relocations only.
// Tabu stamps are bits TB[m] over vehicles, set when a mission leaves a vehicle and cleared
// by a ring of the last `tenure` moves. All moves of entry (v, m) put m on v and share the
// stamp of (m, v), so the least key of a tabu entry aspires if any of its moves does. Swaps
// left out because y is tabu on v(m) can only be applied by aspiration: a new column takes
// its own into account, and TB's companion R[m] keeps a lower bound of their deltas; when
// the bound aspires (rarely), the mission's swaps are evaluated again. When the stamp (y, u)
// expires, node y is evaluated against the missions of u, whose entries (v(y), m) then
// count the swap.
//
// Each CTA keeps the tables of its own slice of the missions (M / CTAs) and the whole
// schedule. Lanes hold missions: 32, or with short slices gm = 2^gm_log of them and 32 / gm
// nodes or vehicles side by side. Warps take units: some nodes of a changed route against a
// block of missions, 32 row entries, or some vehicles' entries of a block. Keys are merged by
// minima, which commute, so results do not depend on the split.

struct CTab32 {  // the matrix's element
  static constexpr int kBytes = 4;
  using T = int32_t;
};
struct CTab16 {
  static constexpr int kBytes = 2;
  using T = int16_t;
};

// Travel time at a byte offset from the start of the matrix (which is at the start of
// dynamic shared memory).
template <class TT>
__device__ __forceinline__ int tmat(int off) {
  return *reinterpret_cast<const typename TT::T*>(reinterpret_cast<const char*>(g_smem) + off);
}

// The matrix through the interface the prologue's helpers use (rows are type * L + location).
template <class TT>
struct CarryTab {
  int cmat, eloc, sloc, Mp, L, RB;  // RB: bytes per row
  __device__ __forceinline__ int row(int tyl, int loc) const { return tyl + loc; }
  __device__ __forceinline__ int a(int r, int m) const {
    return tmat<TT>(r * RB + g_smem[sloc + m] * TT::kBytes) + g_smem[cmat + (r >= L ? Mp : 0) + m];
  }
  __device__ __forceinline__ int b(int r, int m) const {
    const int tyl = r >= L ? L : 0;
    return tmat<TT>((tyl + g_smem[eloc + m]) * RB + (r - tyl) * TT::kBytes);
  }
};

// Records of node t, eight words:
//   {node word, matrix row (byte offset) of the previous node's end, matrix column (bytes)
//    of the next node's start, slot cost | leg into t, removal delta, column of t's start,
//    row of t's end in layer 0}
// D4 (arrive-by times): {departure from the previous node, latest arrival that keeps t's
// time, the same at the next node, removal link ok}.
// VR of a vehicle: {flight minus the duty cap, byte offset of its layer, offset of its
// layer's own legs, 0}.
struct CarryLinks {  // node words and predecessors
  int rec, prv_off;
  __device__ __forceinline__ int32_t& nv(int t) const { return g_smem[rec + 8 * t]; }
  __device__ __forceinline__ int32_t* prv() const { return g_smem + prv_off; }
};

struct CarryCtx {
  int M, N, Mp, horizon, lam;
  int RB, LB;     // bytes of a matrix row, of a layer
  int rec, d4, vr, cmat, wm, tb, kt, it, rb;  // word offsets: records, vehicle records, tables, bounds
  int Sp, S, m0;  // the slice: missions m0 .. m0 + S - 1, row stride Sp (odd)
  int VW;         // 32-bit words of a vehicle set
  uint32_t mul, inv, add;  // detour keys: (detour + add) * mul + y (see unpack_detour)
};

__device__ __forceinline__ int4 ld4(int off) { return *reinterpret_cast<const int4*>(g_smem + off); }
__device__ __forceinline__ uint64_t* kentry(const CarryCtx& c, int v, int i) {
  return reinterpret_cast<uint64_t*>(g_smem + c.kt) + v * c.Sp + i;
}
__device__ __forceinline__ uint32_t* ientry(const CarryCtx& c, int v, int i) {
  return reinterpret_cast<uint32_t*>(g_smem + c.it) + v * c.Sp + i;
}
// word of the vehicle set of mission m that holds vehicle v
__device__ __forceinline__ uint32_t tb_word(const CarryCtx& c, int m, int v) {
  return static_cast<uint32_t>(g_smem[c.tb + (v >> 5) * c.Mp + m]);
}

// Detour keys order by (detour, y): detour + maxT (at least 0, at most 4 maxT) times mul plus
// y. mul is a power of two, or N for the few instances whose times are too long for that (the
// overflow guard bounds 4 maxT N below 2^32). inv = floor(2^32 / mul) gives the quotient or one
// less.
constexpr uint32_t kNoDetour = 0xFFFFFFFFu;
__device__ __forceinline__ void unpack_detour(const CarryCtx& c, uint32_t k, int& ins, int& y) {
  uint32_t d = __umulhi(k, c.inv), r = k - d * c.mul;
  const bool up = r >= c.mul;
  d = up ? d + 1u : d;
  r = up ? r - c.mul : r;
  ins = static_cast<int>(d - c.add);
  y = static_cast<int>(r);
}

template <bool DL, class TT>
__device__ __forceinline__ void carry_record(const Smem& sm, const CarryCtx& c, int t, int nx, int pv, int vw) {
  const int plane = vw_plane(vw);
  const int lay = plane * c.LB, own = c.cmat + plane * c.Mp;
  const int rowE = lay + sm.eloc[pv] * c.RB, eR = sm.eloc[t] * c.RB;
  const int sB = sm.sloc[t] * TT::kBytes, snB = sm.sloc[nx] * TT::kBytes;
  const bool mission = t < c.M;
  const int ct = mission ? g_smem[own + t] : 0;
  int leg = tmat<TT>(rowE + sB);
  const int out = tmat<TT>(lay + eR + snB);
  int lnk = tmat<TT>(rowE + snB);
  if (!mission && pv == t) leg = 0;
  if (nx >= c.M && pv >= c.M) lnk = 0;
  const int slot = mission ? leg + ct + out : 0;
  *reinterpret_cast<int4*>(g_smem + c.rec + 8 * t) = make_int4(nx | (vw << 13), rowE, snB, slot);
  *reinterpret_cast<int4*>(g_smem + c.rec + 8 * t + 4) = make_int4(leg, mission ? lnk - slot : 0, sB, eR);
  if (DL) {
    int4 d = make_int4(pv < c.M ? sm.wm[pv] : 0, c.horizon, 0, 1);
    if (mission) {
      d.y = sm.wm[t] - ct;
      d.z = nx < c.M ? sm.wm[nx] - g_smem[own + nx] : c.horizon;
      d.w = d.x + lnk <= d.z ? 1 : 0;
    }
    *reinterpret_cast<int4*>(g_smem + c.d4 + 4 * t) = d;
  }
}

// No move: above every delta (they stay below 2^31 - 1).
constexpr int kNoDelta = INT32_MAX;
__device__ __forceinline__ uint64_t move_key(int delta, uint32_t id) {
  return pack_key(delta, delta == kNoDelta ? 0xFFFFFFFFu : id);
}

// Delta of the relocation that a detour key into a route of flight fv stands for (kNoDelta
// when there is none), and the node y it goes before. rp: the delta of the mission's own route
// when it leaves; rem: the change of that route's flight; can: it may leave (or, same: move
// within its own route).
template <bool PEN>
__device__ __forceinline__ int reloc_delta(const CarryCtx& c, int rem, int rp, bool can, bool same, int fv, uint32_t k,
                                           int& y) {
  int ins;
  unpack_detour(c, k, ins, y);
  const int g = same ? ins + rem : ins;  // change of the route's flight
  bool ok = (k != kNoDetour) & can;
  int delta;
  if (PEN) {
    delta = (same ? 0 : rp) + g + c.lam * (pos0(fv + g) - pos0(fv));
  } else {
    delta = rem + ins;
    ok = ok & (fv + g <= 0);
  }
  return ok ? delta : kNoDelta;
}

// A mission as the lane's own side of its moves, against one vehicle v.
struct Mine {
  int m, next, rowE, snB, slot, rem, sB, rD;  // rD: row of its end in v's layer
  int vm, layM, ownM, fm, cm, fv, p0;         // p0: pos0(fv) + pos0(fm)
  int rp;
  uint32_t vbit;   // bit of v(m) in a vehicle set
  int hmask;       // heli-only bit of a node word if v(m) is a plane
  int w;
  int4 d;
  bool same, tabu, barred, can;
};

template <bool PEN, bool DL>
__device__ __forceinline__ Mine load_mine(const CarryCtx& c, int m, int v) {
  Mine r;
  const int4 x = ld4(c.rec + 8 * m), q = ld4(c.rec + 8 * m + 4);
  const int4 vv = ld4(c.vr + 4 * v);
  r.m = m;
  r.vm = nv_veh(x.x);
  const int4 vo = ld4(c.vr + 4 * r.vm);
  const uint32_t set = tb_word(c, m, v);
  r.cm = g_smem[vv.z + m];
  if (DL) {
    r.d = ld4(c.d4 + 4 * m);
    r.w = g_smem[c.wm + m];
  }
  r.next = nv_next(x.x);
  r.rowE = x.y;
  r.snB = x.z;
  r.slot = x.w;
  r.rem = q.y;
  r.sB = q.z;
  r.rD = vv.y + q.w;
  r.layM = vo.y;
  r.ownM = vo.z;
  r.fm = vo.x;
  r.fv = vv.x;
  r.same = v == r.vm;
  r.tabu = (set >> (v & 31)) & 1u;
  r.barred = vv.y != 0 && ((x.x >> 24) & 1);
  r.vbit = 1u << (r.vm & 31);
  r.hmask = vo.y != 0 ? 1 << 24 : 0;
  const int pm = pos0(r.fm);
  r.p0 = pos0(r.fv) + pm;
  r.can = DL ? r.d.w != 0 : true;
  if (PEN) {
    r.rp = r.rem + c.lam * (pos0(r.fm + r.rem) - pm);
  } else {
    r.rp = 0;
    r.can = r.can & (r.same | (r.fm + r.rem <= 0));
  }
  return r;
}

constexpr int64_t kNoSwap = INT64_MAX;
// What the lane's mission reads for node y, all of it for every node (of a route's end too),
// so that two nodes' loads can go side by side: with 8 or 16 warps an SM a node is a chain of
// dependent loads. One node at a time, with branches: 193 missions on 3 vehicles, alone on 256
// threads, 46.2 ms for 2,000 iterations; without branches 40.3; two at a time 38.1 (a branch around
// an odd last one, or a loop of its own for short slices, took it back: the larger body, and the two
// evaluations no longer interleaved).
struct NodeTimes {
  int4 x, q, dy;
  int a, b, b2, a3, b3, own, wy;
  uint32_t set;
};
template <bool DL, class TT>
__device__ __forceinline__ NodeTimes load_node(const CarryCtx& c, const Mine& r, int y) {
  NodeTimes t;
  t.x = ld4(c.rec + 8 * y);
  t.q = ld4(c.rec + 8 * y + 4);
  if (DL) {
    t.dy = ld4(c.d4 + 4 * y);
    t.wy = g_smem[c.wm + y];
  }
  t.own = g_smem[r.ownM + y];
  t.set = static_cast<uint32_t>(g_smem[c.tb + (c.VW == 1 ? 0 : (r.vm >> 5) * c.Mp) + y]);
  t.a = tmat<TT>(t.x.y + r.sB) + r.cm;
  t.b = tmat<TT>(r.rD + t.q.z);
  t.b2 = tmat<TT>(r.rD + t.x.z);
  t.a3 = tmat<TT>(r.rowE + t.q.z) + t.own;
  t.b3 = tmat<TT>(r.layM + t.q.w + r.snB);
  return t;
}
// The lane's mission against node y of the vehicle: the detour key of m before y is taken
// into ki, (delta, y) of the swap of m and y into wk, or into wt when y is tabu on v(m) (for a
// given m, swap ids order as y).
template <bool PEN, bool DL, class TT>
__device__ __forceinline__ void eval_node(const CarryCtx& c, const Mine& r, int y, const NodeTimes& n, uint32_t& ki,
                                          int64_t& wk, int64_t& wt) {
  const int a = n.a, b = n.b;
  const bool mfirst = y == r.next, self = y == r.m;
  {
    const uint32_t k = static_cast<uint32_t>(a + b - n.q.x + static_cast<int>(c.add)) * c.mul + static_cast<uint32_t>(y);
    bool ok = !mfirst & !self;
    if (DL) ok = ok & (n.dy.x + a <= r.w) & (r.w + b <= n.dy.y);
    ki = ok & (k < ki) ? k : ki;
  }
  int da = a + n.b2 - n.x.w, db = n.a3 + n.b3 - r.slot;
  // Neighbours fly straight from one to the other, in the other direction than before: with
  // f before s, the new cost is (prev f -> s) + (s -> f) + (f -> next s) against both slots,
  // which count the old leg (f -> s) twice.
  const bool yfirst = nv_next(n.x.x) == r.m;
  int am = a, ay = n.a3;  // flights into m and y in their new places
  if ((mfirst | yfirst) & (y < c.M)) {
    const int back = tmat<TT>(r.layM + n.q.w + r.sB);  // from y's delivery to m's pickup
    if (mfirst) {
      am = back + r.cm;
      da = am + n.b2 - n.x.w;
      db = n.a3 + b - r.slot;
    } else {
      ay = b + n.own;
      da = a + back - n.x.w;
      db = ay + n.b3 - r.slot;
    }
  }
  const int d = da + db;
  int delta;
  bool ok = (y < c.M) & !self & !(n.x.x & r.hmask);
  if (PEN) {
    const int gv = r.same ? d : da, gm = r.same ? 0 : db;
    delta = d + c.lam * (pos0(r.fv + gv) + pos0(r.fm + gm) - r.p0);
  } else {
    delta = d;
    ok = ok & (r.same ? r.fv + d <= 0 : ((r.fv + da <= 0) & (r.fm + db <= 0)));
  }
  if (DL) {
    const bool l1 = (mfirst ? n.wy : n.dy.x) + am <= r.w;
    const bool l2 = yfirst | (r.w + n.b2 <= n.dy.z);
    const bool l3 = (yfirst ? r.w : r.d.x) + ay <= n.wy;
    const bool l4 = mfirst | (n.wy + n.b3 <= r.d.z);
    ok = ok & l1 & l2 & l3 & l4;
  }
  const int64_t k = (static_cast<int64_t>(delta) << 32) | y;
  const bool barred = (n.set & r.vbit) != 0;
  wk = ok & !barred & (k < wk) ? k : wk;
  wt = ok & barred & (k < wt) ? k : wt;
}

// The key of the lane's least swap.
__device__ __forceinline__ uint64_t swap_key(int m, int64_t wk) {
  const int y = static_cast<int>(wk & 0xFFFFFFFF);
  const int m1 = m < y ? m : y, m2 = m < y ? y : m;
  const uint64_t k = pack_key(static_cast<int>(wk >> 32),
                              kSwapBit | (static_cast<uint32_t>(m1) << kIdShift) | static_cast<uint32_t>(m2));
  return wk == kNoSwap ? kNoKey : k;
}

// The entry (v, m) from the least detour and the least swap of a set of v's nodes (of equal
// deltas the relocation has the smaller id). The caller leaves barred missions out.
template <bool PEN>
__device__ __forceinline__ uint64_t entry_key(const CarryCtx& c, const Mine& r, uint32_t ki, int64_t wk) {
  int y;
  const int dr = reloc_delta<PEN>(c, r.rem, r.rp, r.can, r.same, r.fv, ki, y);
  const int ds = static_cast<int>(wk >> 32), ys = static_cast<int>(wk & 0xFFFFFFFF);
  const bool swap = ds < dr;
  const int other = swap ? ys : y;
  const int m1 = swap ? min(r.m, ys) : r.m, m2 = swap ? max(r.m, ys) : other;
  const uint32_t id = (static_cast<uint32_t>(m1) << kIdShift) | static_cast<uint32_t>(m2) | (swap ? kSwapBit : 0u);
  return move_key(swap ? ds : dr, id);
}

// The least swap of mission x with any mission, tabu or not (one warp); its bound becomes the
// least delta of those with missions tabu on v(x). c by value: its fields stay in registers.
template <bool PEN, bool DL, class TT>
__device__ __noinline__ uint64_t all_swaps(const CarryCtx c, int x) {
  const int lane = threadIdx.x & 31;
  uint64_t k = kNoKey;
  int64_t least = kNoSwap;
  for (int y0 = 0; y0 < c.M; y0 += 32) {
    const int y = y0 + lane;
    if (y >= c.M) continue;
    const Mine r = load_mine<PEN, DL>(c, x, nv_veh(g_smem[c.rec + 8 * y]));
    uint32_t unused = kNoDetour;
    int64_t wk = kNoSwap, wt = kNoSwap;
    if (!r.barred) eval_node<PEN, DL, TT>(c, r, y, load_node<DL, TT>(c, r, y), unused, wk, wt);
    k = min_u64(k, min_u64(swap_key(x, wk), swap_key(x, wt)));
    least = wt < least ? wt : least;
  }
  const int bound = __reduce_min_sync(0xffffffffu, static_cast<int>(least >> 32));
  if (lane == 0) g_smem[c.rb + x - c.m0] = bound;
  return k;
}

// One complete search of the instance in P, as solve_one, with carried move values; lay is a
// carry layout.
template <bool PEN, bool DL, class TT>
__device__ __forceinline__ void carry_solve(const KParams& P, const Layout& lay, const int C, const int rank) {
  const bool lead = rank == 0;
  const Smem sm = carve(lay);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  const int M = P.M, V = P.V, N = P.M + P.V, L = P.L, Mp = lay.Mp, nt = P.nt;
  Ctx c0;
  c0.M = M;
  c0.V = V;
  c0.N = N;
  c0.L = L;
  c0.Mp = Mp;
  c0.cap = P.cap;
  c0.horizon = P.horizon;
  c0.lam = P.lambda;
  c0.heli = 1;
  CarryCtx c;
  c.M = M;
  c.N = N;
  c.Mp = Mp;
  c.horizon = P.horizon;
  c.lam = P.lambda;
  c.RB = lay.Ls * TT::kBytes;
  c.LB = L * c.RB;
  c.rec = lay.rec;
  c.d4 = lay.d4;
  c.vr = lay.vr;
  c.cmat = lay.cmat;
  c.wm = lay.wm;
  c.tb = lay.tb;
  c.kt = lay.ktab;
  c.it = lay.itab;
  c.rb = lay.bound;
  c.Sp = lay.Sp;
  c.VW = lay.VW;
  const int slice = lay.S;  // missions per CTA
  c.m0 = rank * slice < M ? rank * slice : M;
  c.S = M - c.m0 < slice ? M - c.m0 : slice;
  int status = ASCHED_OK;

  // ---- prologue: statics, the matrix, its checks
  if (tid < 16) sm.misc[tid] = 0;
  __syncthreads();
  int any_heli = 0;
  int bad = load_statics(P, sm, Mp, round_up(N + 1, 4), any_heli);
  int maxT = 0;
  if (TT::kBytes == 4) {
    for (int i = tid; i < nt * L * L; i += nthr) {
      const int x = gin(P.travel + i);
      bad |= x < 0;
      maxT = x > maxT ? x : maxT;
      const int r = i / L;
      g_smem[r * lay.Ls + (i - r * L)] = x;
    }
  }
  if (__syncthreads_or(bad)) status = ASCHED_E_INVALID;
  if (TT::kBytes == 2 && status == ASCHED_OK) {
    int tbad = 0;
    const bool timed_out = stage_matrix16(P, lay, C, tbad, maxT);
    if (__syncthreads_or(tbad)) status = ASCHED_E_INVALID;
    if (timed_out) status = ASCHED_E_TIMEOUT;  // the same in every CTA of the cluster
  }
  maxT = __reduce_max_sync(0xffffffffu, maxT);
  if (lane == 0) atomicMax(&sm.misc[MISC_MAXT], maxT);
  __syncthreads();
  maxT = sm.misc[MISC_MAXT];
  if (lay.big && status == ASCHED_OK && maxT > 32767) status = ASCHED_E_TOO_LARGE;
  if (status == ASCHED_OK) {
    // 2 (2M + V + 2) maxT (1 + lambda) < 2^31 keeps every int32 sum in range.
    const double bound = 2.0 * (2.0 * M + V + 2.0) * static_cast<double>(maxT) *
                         (1.0 + (PEN ? static_cast<double>(c.lam) : 0.0));
    if (!(bound < 2147483648.0)) status = ASCHED_E_OVERFLOW_GUARD;
  }
  // a detour lies in [-maxT, 3 maxT]; the shifted key must stay below all ones (no gap)
  c.add = static_cast<uint32_t>(maxT);
  const int shift = 32 - __clz(N > 1 ? N - 1 : 1);
  c.mul = ((4ull * maxT + 1ull) << shift) < 0xFFFFFFFFull ? 1u << shift : static_cast<uint32_t>(N);
  c.inv = c.mul > 1u ? static_cast<uint32_t>(0x100000000ull / c.mul) : 0xFFFFFFFFu;

  const CarryLinks S0{lay.rec, lay.prv};
  CarryTab<TT> tb;
  tb.cmat = lay.cmat;
  tb.eloc = lay.eloc;
  tb.sloc = lay.sloc;
  tb.Mp = Mp;
  tb.L = L;
  tb.RB = c.RB;
  if (status == ASCHED_OK) {
    for (int i = tid; i < nt * Mp; i += nthr) {
      const int t = i / Mp, m = i - t * Mp;
      sm.cmat[i] = m < M ? tmat<TT>(t * c.LB + sm.sloc[m] * c.RB + sm.eloc[m] * TT::kBytes) : 0;
    }
    for (int v = tid; v < V; v += nthr) {
      S0.nv(M + v) = (M + v) | ((v | ((sm.vtype[v] != 0 ? 1 : 0) << 10)) << 13);
      S0.prv()[M + v] = M + v;
    }
  }
  __syncthreads();
  if (status == ASCHED_OK) status = initial_schedule<PEN, DL>(P, sm, tb, S0, c0);
  int Z = 0;
  if (status == ASCHED_OK) {
    const bool ok = start_records<PEN, DL>(sm, tb, S0, c0, [&](int t, int nx, int pv, int vw, int f) {
      carry_record<DL, TT>(sm, c, t, nx, pv, vw);
      if (t >= M)
        *reinterpret_cast<int4*>(g_smem + c.vr + 4 * (t - M)) =
            make_int4(f - P.cap, vw_plane(vw) * c.LB, c.cmat + vw_plane(vw) * Mp, 0);
    });
    if (!ok) status = ASCHED_E_INFEASIBLE_INIT;
    for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S0.nv(t));
    for (int i = tid; i < 2 * kMaxCluster; i += nthr) sm.slots()[i] = 0;
    if (tid < 2) sm.gkey()[tid] = 0;
    __syncthreads();
    Z = sm.misc[MISC_Z0];
  }

  int zbest = Z, best_it = -1, it = 0;
  const bool looped = status == ASCHED_OK;  // uniform over the cluster
  if (looped) {
    if (C > 1) cluster_sync_all();
    // ---- tables of the start schedule. The prologue's scratch (sm.gfl etc.) ends here.
    for (int i = tid; i < c.VW * Mp; i += nthr) g_smem[c.tb + i] = 0;
    for (int i = tid; i < 2 * P.tenure; i += nthr) g_smem[lay.ring + i] = -1;
    if (tid < 8) g_smem[lay.ccnt + tid] = 0;
    if (tid < 4) g_smem[lay.expired + tid] = -1;
    for (int i = tid; i < c.S; i += nthr) g_smem[c.rb + i] = INT32_MAX;
    __syncthreads();
    const int gl = lay.gm_log, gm = 1 << gl, subs = 32 >> gl, sub = lane >> gl;
    const int nblk = (c.S + gm - 1) >> gl;  // blocks of missions (several only with gm = 32)
    for (int u = P.iterations > 0 ? warp : nblk * V; u < nblk * V; u += nwarps) {
      const int blk = u % nblk, v = u / nblk;
      const int i = blk * 32 + (lane & (gm - 1));
      const Mine r = load_mine<PEN, DL>(c, c.m0 + (i < c.S ? i : 0), v);
      uint32_t ki = kNoDetour;
      int64_t wk = kNoSwap, wt = kNoSwap;
      for (int y = nv_next(S0.nv(M + v));; y = nv_next(S0.nv(y))) {
        eval_node<PEN, DL, TT>(c, r, y, load_node<DL, TT>(c, r, y), ki, wk, wt);
        if (y >= M) break;
      }
      if (r.barred) {
        ki = kNoDetour;
        wk = kNoSwap;
      }
      if (i < c.S && sub == 0) {
        *ientry(c, v, i) = ki;
        *kentry(c, v, i) = entry_key<PEN>(c, r, ki, wk);
      }
    }
    __syncthreads();

    // Column units: 2^sh nodes of a changed route against one block of missions, at least
    // 2^lay.ulog of them and at most lay.ucap units. Their lanes take entries' deltas by a
    // 32-bit atomic minimum and leave their keys in pk; the apply step, when the deltas are
    // final, takes the least id among the keys that have it (64-bit shared-memory minima are
    // compare-and-swap loops).
    uint64_t* const pk = reinterpret_cast<uint64_t*>(g_smem + lay.pkey);
    const int vspan = lay.kv * subs;
    const int PV = (V + vspan - 1) / vspan;  // scan units per block
    const uint32_t binv = nblk > 1 ? 0xFFFFFFFFu / static_cast<uint32_t>(nblk) + 1u : 0u;  // the same for blocks
    const uint32_t vinv = 0xFFFFFFFFu / static_cast<uint32_t>(V) + 1u;  // x / V = umulhi(x, vinv) for V > 1, small x
    uint16_t* const listA = reinterpret_cast<uint16_t*>(g_smem + lay.list);
    uint16_t* const listB = listA + round_up(N, 8);
    uint16_t* const rows = reinterpret_cast<uint16_t*>(g_smem + lay.rows);
    const int stop_word = lay.misc + MISC_STOP;
    const int wlist = nwarps >= 4 ? 2 : 1;  // first warp that lists the changed routes' nodes
    int va = -1, vb = -1;  // routes the last move changed
    int rslot = 0;         // ring slot of this iteration (it mod tenure)
    bool copy_best = false;
    const int iters = P.iterations;
    for (it = 0; it < iters; ++it) {
      const int zrel = zbest - Z;
      const int par = (it & 1) * 4, ppar = 4 - par;  // counters written by this iteration's apply, by the last one's
      int PA = 0, PB = 0, sh = lay.ulog;
      uint64_t key = kNoKey;
      if (nblk > 0) {
        const int4 cn = ld4(lay.ccnt + ppar);  // nodes of va's and vb's routes, unused, rows
        const int2 ex = *reinterpret_cast<const int2*>(g_smem + lay.expired);  // stamps that expired
        const int nA = cn.x, nB = cn.y;
        PA = (nA + (1 << sh) - 1) >> sh;
        PB = (nB + (1 << sh) - 1) >> sh;
        while ((PA + PB) * nblk > lay.ucap) {
          ++sh;
          PA = (nA + (1 << sh) - 1) >> sh;
          PB = (nB + (1 << sh) - 1) >> sh;
        }
        // units: columns, expired stamps, rows, entries of the other missions
        // rows: with one CTA the missions of both lists, else those listed for this CTA's slice
        const int nE = (ex.x >= 0) + (ex.y >= 0), nRV = (C > 1 ? cn.w : nA + nB) * V;
        const int e1 = (PA + PB) * nblk, e2 = e1 + nE * nblk, e3 = e2 + ((nRV + 31) >> 5), e4 = e3 + PV * nblk;
        for (int u = warp; u < e4; u += nwarps) {
          if (u < e2) {
            // ---- nodes of a changed route, or a mission whose stamp expired, against a block
            const bool column = u < e1;
            const int uu = column ? u : u - e1;
            const int pc = nblk == 1 ? uu : static_cast<int>(__umulhi(static_cast<uint32_t>(uu), binv));
            const int i = (uu - pc * nblk) * 32 + (lane & (gm - 1));
            const bool act = i < c.S;
            const int m = c.m0 + (act ? i : 0);
            const bool first = pc < PA;
            const int e = pc == 0 && ex.x >= 0 ? ex.x : ex.y;
            const int v = column ? (first ? va : vb) : nv_veh(g_smem[c.rec + 8 * (e >> 10)]);
            const Mine r = load_mine<PEN, DL>(c, m, v);
            uint32_t ki = kNoDetour;
            int64_t wk = kNoSwap, wt = kNoSwap;
            if (column) {
              const uint16_t* list = first ? listA : listB;
              const int n = first ? nA : nB;
              const int k0 = (first ? pc : pc - PA) << sh, k1 = k0 + (1 << sh) < n ? k0 + (1 << sh) : n;
              for (int k = k0 + sub; k < k1; k += 2 * subs) {  // two nodes' loads side by side (an odd last one twice)
                const int y0 = list[k], y1 = list[k + subs < k1 ? k + subs : k];
                const NodeTimes t0 = load_node<DL, TT>(c, r, y0), t1 = load_node<DL, TT>(c, r, y1);
                eval_node<PEN, DL, TT>(c, r, y0, t0, ki, wk, wt);
                eval_node<PEN, DL, TT>(c, r, y1, t1, ki, wk, wt);
              }
            } else if (sub == 0 && r.vm == (e & 0x3FF)) {
              eval_node<PEN, DL, TT>(c, r, e >> 10, load_node<DL, TT>(c, r, e >> 10), ki, wk, wt);
              ki = kNoDetour;
            }
            if (r.barred | !act) {
              ki = kNoDetour;
              wk = wt = kNoSwap;
            }
            const uint64_t ek = entry_key<PEN>(c, r, ki, wk);
            const bool on = !r.tabu | (key_delta(ek) < zrel);
            key = on & (ek < key) ? ek : key;
            if (wt != kNoSwap) {  // swaps with missions tabu on v(m)
              const int d = static_cast<int>(wt >> 32);
              if (d < zrel) key = min_u64(key, swap_key(m, wt));
              atomicMin(&g_smem[c.rb + i], d);
            }
            const int at = v * c.Sp + i;
            if (column) {
              pk[u * 32 + lane] = ek;
              if (act) {
                atomicMin(reinterpret_cast<uint32_t*>(g_smem) + c.it + at, ki);
                atomicMin(reinterpret_cast<uint32_t*>(g_smem) + c.kt + 2 * at + 1, static_cast<uint32_t>(ek >> 32));
              }
            } else if (ek != kNoKey) {
              atomicMin(reinterpret_cast<unsigned long long*>(g_smem + c.kt) + at, ek);
            }
          } else if (u < e3) {
            // ---- rows of missions whose route changed: relocations into the other routes
            const int x = (u - e2) * 32 + lane;
            const int k = V > 1 ? static_cast<int>(__umulhi(static_cast<uint32_t>(x), vinv)) : x;
            const int v = x - k * V;
            const int m = x < nRV ? (C > 1 ? rows[k] : (k < nA ? listA[k] : listB[k - nA])) : M;
            if (m < M && v != va && v != vb) {
              const int i = m - c.m0;
              const int vm = nv_veh(g_smem[c.rec + 8 * m]), rem = g_smem[c.rec + 8 * m + 5];
              const int fm = g_smem[c.vr + 4 * vm], fv = g_smem[c.vr + 4 * v];
              const uint32_t ki = *ientry(c, v, i);
              const bool tabu = (tb_word(c, m, v) >> (v & 31)) & 1u;
              const int rp = PEN ? rem + c.lam * (pos0(fm + rem) - pos0(fm)) : 0;
              bool can = PEN || fm + rem <= 0;
              if (DL) can = can & (g_smem[c.d4 + 4 * m + 3] != 0);
              int y;
              const int d = reloc_delta<PEN>(c, rem, rp, can, false, fv, ki, y);
              const uint64_t ek = move_key(d, (static_cast<uint32_t>(m) << kIdShift) | static_cast<uint32_t>(y));
              *kentry(c, v, i) = ek;
              key = (!tabu | (d < zrel)) & (ek < key) ? ek : key;
            }
          } else {
            // ---- entries of the other missions
            const int uu = u - e3;
            const int ch = nblk == 1 ? uu : static_cast<int>(__umulhi(static_cast<uint32_t>(uu), binv));
            const int i = (uu - ch * nblk) * 32 + (lane & (gm - 1));
            const int m = c.m0 + (i < c.S ? i : 0);
            const int vm = nv_veh(g_smem[c.rec + 8 * m]);
            const bool on = i < c.S && vm != va && vm != vb;
            const int v0 = ch * vspan + sub;
            const int v1 = on ? ((ch + 1) * vspan < V ? (ch + 1) * vspan : V) : 0;
            const uint64_t* kp = reinterpret_cast<const uint64_t*>(g_smem + c.kt) + v0 * c.Sp + (i < c.S ? i : 0);
            const int kstep = subs * c.Sp;
            uint32_t set = static_cast<uint32_t>(g_smem[c.tb + (v0 >> 5) * Mp + m]);
            int word = v0 >> 5;
            for (int v = v0; v < v1; v += 4 * subs) {  // four entries at a time, loads first
              uint64_t k[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) k[j] = v + j * subs < v1 ? kp[j * kstep] : kNoKey;
              kp += 4 * kstep;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int vj = v + j * subs;
                if ((vj >> 5) != word && vj < v1) {
                  word = vj >> 5;
                  set = static_cast<uint32_t>(g_smem[c.tb + word * Mp + m]);
                }
                const bool ok = (vj != va) & (vj != vb) & (!((set >> (vj & 31)) & 1u) | (key_delta(k[j]) < zrel));
                key = ok & (k[j] < key) ? k[j] : key;
              }
            }
            // swaps with missions tabu on v(m), where their bound aspires
            uint32_t again = __ballot_sync(0xffffffffu, ch == 0 && sub == 0 && i < c.S && g_smem[c.rb + i] < zrel);
            while (again) {
              const int at = __ffs(again) - 1;
              again &= again - 1;
              const int x = __shfl_sync(0xffffffffu, m, at);
              const uint64_t k = all_swaps<PEN, DL, TT>(c, x);
              if (key_delta(k) < zrel) key = min_u64(key, k);
            }
          }
        }
      }
      if (copy_best) {
        for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S0.nv(t));
      }
      if (tid < 4) g_smem[lay.ccnt + par + tid] = 0;
      if (warp == nwarps - 1 && P.tenure > 0) {
        // stamps that expire after this iteration: the ring slot's, unless set again since
        const int o0 = g_smem[lay.ring + 2 * rslot], o1 = g_smem[lay.ring + 2 * rslot + 1];
        bool again0 = false, again1 = false;
        for (int k = lane; k < 2 * P.tenure; k += 32) {
          const int e = g_smem[lay.ring + k];
          again0 |= ((k >> 1) != rslot) & (e == o0);
          again1 |= ((k >> 1) != rslot) & (e == o1);
        }
        const uint32_t a0 = __ballot_sync(0xffffffffu, again0), a1 = __ballot_sync(0xffffffffu, again1);
        if (lane < 2) g_smem[lay.expired + 2 + lane] = lane == 0 ? (a0 ? -1 : o0) : (a1 ? -1 : o1);
      }
      key = warp_min_key(key);
      if (lane == 0) sm.warpkey()[warp] = key;
      __syncthreads();
      uint64_t gk = warp_min_key(lane < nwarps ? sm.warpkey()[lane] : kNoKey);
      bool timed_out = false;
      if (C > 1) gk = exchange_keys(P, sm, C, rank, 1, 0, it, gk, timed_out);
      const bool bad_key = !timed_out && !key_names_nodes(gk, M, N);
      const bool go = !timed_out && !bad_key;
      const bool moved = go && gk != kNoKey;
      const int pva = va, pvb = vb;  // the columns whose partial minima are put together below
      const uint32_t id = static_cast<uint32_t>(gk);
      const bool is_swap = moved && (id & kSwapBit) != 0;
      // relocation: mission n1 before node n2; swap: missions n1, n2
      const int n1 = moved ? static_cast<int>((id >> kIdShift) & kIdMask) : 0;
      const int n2 = moved ? static_cast<int>(id & kIdMask) : 0;
      const int nv1 = S0.nv(n1), nv2 = S0.nv(n2);
      va = moved ? nv_veh(nv1) : -1;
      vb = moved ? nv_veh(nv2) : -1;
      copy_best = false;
      if (moved) {
        Z += key_delta(gk);
        if (Z < zbest) {
          zbest = Z;
          best_it = it;
          copy_best = true;
        }
      }
      // Every warp comes to barrier 1 once per iteration: warp 0 waits there, before it rewrites
      // the move's nodes, for the others to have read them.
      if (warp == 0) {
        // ---- the at most six relinked nodes, one per lane
        const int x1 = nv_next(nv1), x2 = nv_next(nv2);
        const int p1 = S0.prv()[n1], p2 = S0.prv()[n2];
        int t = n1;
        if (lane == 1) t = n2;
        if (lane == 2) t = p1;
        if (lane == 3) t = x1;
        if (lane == 4) t = p2;
        if (lane == 5) t = x2;
        const int nvt = S0.nv(t);
        int nx = nv_next(nvt), pv = S0.prv()[t], vw = nv_vw(nvt);
        const int vwa = nv_vw(nv1), vwb = nv_vw(nv2);
        relink(is_swap, n1, n2, p1, x1, p2, x2, vwa, vwb, t, nx, pv, vw);
        named_sync(1, nthr);
        if (moved && lane < 6) {
          carry_record<DL, TT>(sm, c, t, nx, pv, vw);
          S0.prv()[t] = pv;
        }
      } else {
        if (warp == 1 && moved) {
          // ---- the routes' new flights, from the same entries the evaluation used
          const int4 xa = ld4(c.rec + 8 * n1), qa = ld4(c.rec + 8 * n1 + 4);
          const int4 xb = ld4(c.rec + 8 * n2), qb = ld4(c.rec + 8 * n2 + 4);
          const int4 ra = ld4(c.vr + 4 * va), rb = ld4(c.vr + 4 * vb);
          int da, db;
          const int cab = g_smem[rb.z + n1];  // n1's own leg on vb's layer
          if (!is_swap) {
            da = qa.y;
            db = tmat<TT>(xb.y + qa.z) + cab + tmat<TT>(rb.y + qa.w + qb.z) - qb.x;
          } else {
            const bool adjA = nv_next(xa.x) == n2, adjB = nv_next(xb.x) == n1;
            // n2 in n1's place, n1 in n2's place; a neighbour's own ends cancel (see eval_node)
            da = tmat<TT>((adjB ? ra.y + qa.w : xa.y) + qb.z) + g_smem[ra.z + n2] +
                 tmat<TT>(adjA ? ra.y + qa.w + qb.z : ra.y + qb.w + xa.z) - xa.w;
            db = tmat<TT>((adjA ? rb.y + qb.w : xb.y) + qa.z) + cab +
                 tmat<TT>(adjB ? rb.y + qb.w + qa.z : rb.y + qa.w + xb.z) - xb.w;
          }
          if (lane == 0) {
            if (va == vb) {
              g_smem[c.vr + 4 * va] = ra.x + da + db;
            } else {
              g_smem[c.vr + 4 * va] = ra.x + da;
              g_smem[c.vr + 4 * vb] = rb.x + db;
            }
          }
          __syncwarp();
        }
        named_arrive(1, nthr);
        if (moved && warp >= wlist) {
          // ---- the changed routes' nodes (their vehicles after the move), in any order
          for (int t = tid - 32 * wlist; t < N; t += nthr - 32 * wlist) {
            int vt = nv_veh(S0.nv(t));
            if (t == n1) vt = vb;
            if (is_swap && t == n2) vt = va;
            if (vt != va && vt != vb) continue;
            const bool inA = vt == va;
            const int at = atomicAdd(&g_smem[lay.ccnt + par + (inA ? 0 : 1)], 1);
            (inA ? listA : listB)[at] = static_cast<uint16_t>(t);
            const int i = t - c.m0;
            if (t < M && i >= 0 && i < c.S) {
              g_smem[c.rb + i] = INT32_MAX;
              if (C > 1) rows[atomicAdd(&g_smem[lay.ccnt + par + 3], 1)] = static_cast<uint16_t>(t);
            }
          }
        }
        if (go) {
          // ---- this iteration's columns (unless they change again): ids of the least deltas
          for (int u = warp - 1; u < (PA + PB) * nblk; u += nwarps - 1) {
            const int pc = nblk == 1 ? u : static_cast<int>(__umulhi(static_cast<uint32_t>(u), binv));
            const int i = (u - pc * nblk) * 32 + (lane & (gm - 1));
            const int v = pc < PA ? pva : pvb;
            if (i < c.S && v != va && v != vb) {
              const uint64_t k = pk[u * 32 + lane];
              uint32_t* const e = reinterpret_cast<uint32_t*>(kentry(c, v, i));
              if (e[1] == static_cast<uint32_t>(k >> 32)) atomicMin(e, static_cast<uint32_t>(k));
            }
          }
        }
        if (moved) {
          for (int x = nthr - 1 - tid; x < 2 * c.S; x += nthr - 32) {
            const int at = x < c.S ? va * c.Sp + x : vb * c.Sp + x - c.S;
            g_smem[c.it + at] = -1;
            *(reinterpret_cast<uint64_t*>(g_smem + c.kt) + at) = kNoKey;
          }
        }
        if (warp == 1 && go && P.tenure > 0) {
          // ---- stamps: the ring slot's old ones expire, this move's are set
          const int s0 = moved ? (n1 << 10) | va : -1, s1 = is_swap ? (n2 << 10) | vb : -1;
          int e = lane < 2 ? g_smem[lay.expired + 2 + lane] : -1;
          if (lane < 2) {
            if (e == s0 || e == s1) e = -1;
            if (e >= 0) {
              const int x = e >> 10, v = e & 0x3FF;
              atomicAnd(&g_smem[c.tb + (v >> 5) * Mp + x], ~(1 << (v & 31)));
              // x's vehicle; a mission of this move flies on va or vb. A changed route's column
              // counts the swaps of x with v's missions anyway.
              const int vx = nv_veh(S0.nv(x));
              if (moved && (vx == va || vx == vb || v == va || v == vb)) e = -1;
            }
            g_smem[lay.expired + lane] = e;
          } else if (lane < 4) {
            const int s = lane == 2 ? s0 : s1;
            if (s >= 0) atomicOr(&g_smem[c.tb + ((s & 0x3FF) >> 5) * Mp + (s >> 10)], 1 << (s & 31));
            g_smem[lay.ring + 2 * rslot + lane - 2] = s;
          }
        }
      }
      if (++rslot >= P.tenure) rslot = 0;
      if (lead && tid == 0 && !timed_out) {
        if (P.traj_move) P.traj_move[it] = gk == kNoKey ? kNullMove : id;
        if (P.traj_z) P.traj_z[it] = Z;
      }
      if (!go) g_smem[stop_word] = bad_key ? ASCHED_E_INVALID : ASCHED_E_TIMEOUT;
      __syncthreads();
      if (!go || (C > 1 && g_smem[stop_word] != 0)) {
        status = g_smem[stop_word];
        break;
      }
    }
    if (copy_best) {
      for (int t = tid; t < N; t += nthr) sm.best[t] = nv_next(S0.nv(t));
    }
    __syncthreads();
  }

  if (lead && status == ASCHED_OK && P.out_off) status = write_schedule(P, sm, c0);
  if (lead && tid == 0 && P.info) write_info(P.info, status, zbest, best_it, sm.misc[MISC_Z0], Z, it);
  // No CTA may leave while a peer can still write into its shared memory.
  if (C > 1 && looped) cluster_sync_unaligned();
}
