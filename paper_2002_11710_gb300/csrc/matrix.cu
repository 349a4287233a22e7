// Travel-time matrices built on the device from location coordinates (Eq. e1,
// Section 3): for every instance of a batch and every vehicle type t,
//   T[t][i][j] = rint(dist_km(i, j) / speed_kmh[t] * 60)   (integer minutes, half to even)
// with the Haversine distance of Eq. e1 on (latitude, longitude) in degrees, or the
// Euclidean distance on (x, y) kilometres. float64 throughout, as the paper's Python.
//
// The Euclidean path rounds every operation explicitly (no contraction into fused
// multiply-adds), in the order subtract, square, add, square root, divide, multiply, so
// it returns the same integers as any IEEE float64 evaluation of that expression. The
// Haversine path calls the device sine, cosine and arcsine, which may differ from a host
// library in the last bits; the integer result then differs only where the exact time
// lies within a few ulps of a half minute.
//
// Most entries are decided in float32, with float64 only where float32 cannot vouch for
// the integer: rint changes value only at half minutes, so when the float32 time lies
// farther from the nearest half minute than a bound on its error, it rounds to the same
// integer as the float64 expression (whose own error is far smaller).
// Bounds on the float32 time t (every float32 value of a coordinate is off by at most
// 2^-24 of its magnitude):
//   Euclidean  coordinates staged as float32; the differences add at most 2^-24 of the
//              sum of the four magnitudes, then differences, squares, sum, square root
//              and the product with a rounded 60 / speed add below 6 * 2^-24 relative with
//              a correctly rounded root, 10 * 2^-24 with the root as a * rsqrtf(a) (rsqrtf
//              within 2 ulp, CUDA's documented bound, plus one rounded product); screened
//              at 2e-6 t + (60 / speed) 2^-20 S + 1e-6, S the instance's largest |x| + |y|;
//   Haversine  angles staged as float pairs hi + lo (lo = float(v - hi)), so a difference
//              (hi_i - hi_j) + (lo_i - lo_j) is within 2 * 2^-24 of itself plus 2^-47 of
//              the magnitudes. Longitudes more than half a turn apart first take the short
//              way round, and latitudes or longitudes still further apart go to float64, so
//              that the half angle's sine has a condition number below 1 (near a whole turn
//              it has no bound: without this, the small kernel rounded times between the two
//              sides of the date line wrongly at 10 km/h; with it 16,384 Haversine instances
//              of 52 locations take 215 us, 213 before). Small instances: half-angle
//              differences, sinf (2 ulp), squares, cos(phi) staged from float64, sum, square
//              root and asinf (2 ulp) with its condition number below 1.9 for sqrt(a) <= 0.9
//              (larger values go to float64 outright) add below 1.8e-6 relative; screened at
//              8e-6 t + (60 / speed) 2 r 2^-40 (sum of |angles|) + 1e-5. Tiles: own fits of
//              sine (4 * 2^-24) and arcsine (asinf where sqrt(a) > 1/2) and cos(phi) within
//              6 * 2^-24 give 27 * 2^-24 for a and below 2.5e-6 for the time (largest found
//              against 80-bit floats over 14 million pairs, poles and date line among them:
//              8.8e-7, 0.22 of the screen); screened at 4e-6 t + the same rest.
// Times of 2^22 minutes or more also go to float64 (small instances: every entry of an
// instance whose largest possible time, 2 S * 60 / speed or pi r * 60 / speed, is not
// below 2^22, through an infinite tolerance). The float32 time is rounded by adding
// and subtracting 1.5 * 2^23: for 0 <= t < 2^22 the sum lies in [2^23, 2^24), where the
// float32 spacing is 1, so the addition itself rounds t half to even, the integer is the
// sum's low mantissa bits, and t minus the rounded value is exact (Sterbenz), which gives
// the distance to the nearest half minute without a conversion instruction. The float64
// path is the expression above, on the original float64 coordinates. Lanes that need it
// queue (row, column, type) in shared memory, so float64 work runs on full warps and
// follows the number of such entries: small instances one queue per instance, drained
// after the pairs by as many warps as it has entries (one, as a rule); tiles one queue over
// a CTA's whole run. Entries beyond a queue's capacity are computed where they arise.
//
// Both distances are symmetric in every rounded operation (x_i - x_j = -(x_j - x_i)
// exactly, products commute), so each unordered pair is evaluated once and written to
// (i, j) and (j, i). Two kernels share a batch:
//   Small instances (n_types * L^2 + 3 <= kOut words, L <= kSmallLoc: L <= 55 for two
//   types, 78 for one), where a batch holds no others or enough of them to fill the chip (a
//   few among larger ones join the tiles), are built whole in shared memory by 128-thread CTAs, eight per SM, one
//   CTA per instance (grid-stride), with its coordinates staged once.
//   The L (L + 1) / 2 pairs are numbered row by row with row
//   i folded onto row L - 1 - i (L + 1 pairs per folded row), so the threads take
//   consecutive numbers with no idle lanes at row ends. The finished matrices, contiguous
//   in the output, leave by one bulk copy (cp.async.bulk, shared to global) on their
//   16-byte aligned middle and plain stores on the at most 3 + 3 words around it; the
//   next instance is staged while that copy runs and waits only for its reads of shared
//   memory, before its first write of the matrix.
//   Other instances by tiles of 64 x 64 pairs (travel_tiles_kernel).
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "asched.h"
#include "nvtx_range.h"

namespace {

constexpr int kWarps = 8;              // tile CTAs: 8 warps, 4 per SM
constexpr int kTile = 64;              // locations of a tile's side
constexpr int kThreads = kWarps * 32;
constexpr int kTileQueue = 512;        // deferred float64 entries per CTA (tiles)
constexpr int kSmallThreads = 128;     // small-instance CTAs: 4 warps, 8 per SM
constexpr int kSmallLoc = 80;          // locations of an instance built in shared memory
constexpr int kOut = 6144;             // int32 words of that instance's matrices
constexpr int kSmallQueue = 256;       // deferred float64 entries per CTA (small instances)

__host__ __device__ __forceinline__ bool is_small(int L, int nt) {
  return L <= kSmallLoc && nt * L * L + 3 <= kOut;
}

struct MParams {
  int32_t B, nt, metric;
  double speed[2];
  float k32[2];  // float(60 / speed)
  float rel_hav;  // Haversine screen: 8e-6, or infinity if a time may reach 2^22 minutes
  double two_r, deg;
  const int32_t* loc_off;
  const int64_t* travel_off;
  const double* coords;
  int32_t* travel;
  int32_t* status;
};

struct SmallStage {  // 26,816 bytes: with the queue, eight CTAs fit one SM
  float4 hl[kSmallLoc];     // (x hi, y hi, x lo, y lo)
  float cphi[kSmallLoc];    // float(cos(phi))
  double cos64[kSmallLoc];  // cos(phi) in float64, as the definition computes it
  int32_t out[kOut];        // the instance's matrices, offset so that they share the output's 16-byte phase
};
static_assert(offsetof(SmallStage, out) % 16 == 0, "the bulk copy reads out at 16-byte boundaries");
static_assert(kSmallLoc <= kSmallThreads, "one location per thread when staging");

__device__ __forceinline__ double euclid(double xi, double yi, double xj, double yj) {
  const double dx = __dsub_rn(xi, xj), dy = __dsub_rn(yi, yj);
  return __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}

// Eq. e1 with the cosines of both latitudes given (each equals cos(lat * deg) bit for bit).
__device__ __forceinline__ double haversine(double lati, double loni, double latj, double lonj, double ci, double cj,
                                            double two_r, double deg) {
  const double phi_i = __dmul_rn(lati, deg), phi_j = __dmul_rn(latj, deg);
  const double s1 = sin(__dmul_rn(__dsub_rn(phi_i, phi_j), 0.5));
  const double s2 = sin(__dmul_rn(__dsub_rn(__dmul_rn(loni, deg), __dmul_rn(lonj, deg)), 0.5));
  const double a = __dadd_rn(__dmul_rn(s1, s1), __dmul_rn(__dmul_rn(ci, cj), __dmul_rn(s2, s2)));
  const double r = __dsqrt_rn(a);
  return __dmul_rn(two_r, asin(r > 1.0 ? 1.0 : r));  // a NaN stays NaN, as in the definition
}

// The definition in float64: distance, then rint(d / speed * 60). cos64: the staged
// cosines of the latitudes (Haversine, small instances) or NULL.
__device__ __forceinline__ double minutes64(const MParams& P, const double* c, const double* cos64, int i, int j,
                                            int t) {
  const double xi = c[2 * i], yi = c[2 * i + 1], xj = c[2 * j], yj = c[2 * j + 1];
  double d;
  if (P.metric == ASCHED_METRIC_HAVERSINE) {
    const double ci = cos64 ? cos64[i] : cos(__dmul_rn(xi, P.deg));
    const double cj = cos64 ? cos64[j] : cos(__dmul_rn(xj, P.deg));
    d = haversine(xi, yi, xj, yj, ci, cj, P.two_r, P.deg);
  } else {
    d = euclid(xi, yi, xj, yj);
  }
  return rint(__dmul_rn(__ddiv_rn(d, P.speed[t]), 60.0));
}

__device__ __forceinline__ int32_t checked(double m, int& bad) {
  const bool ok = m >= 0.0 && m <= 2147483647.0;  // false for NaN too
  bad |= !ok;
  return ok ? static_cast<int32_t>(m) : 0;
}

// One float32 time t32 >= 0 (or NaN): its integer in v, and whether that integer is certain,
// i.e. t32 lies farther than tol = rel t32 + c from every half minute. t32 < 2^22, or rel is
// infinite (the comparison then fails).
__device__ __forceinline__ bool round_screened_bounded(float t32, float rel, float c, int32_t& v) {
  const float s = __fadd_rn(t32, 12582912.0f);
  const float gap = __fsub_rn(0.5f, fabsf(__fsub_rn(t32, __fsub_rn(s, 12582912.0f))));
  v = __float_as_int(s) - 0x4B400000;
  return gap > __fmaf_rn(rel, t32, c);
}

// Difference of two staged longitudes in radians, (x hi, y hi, x lo, y lo) each. Longitudes
// more than half a turn apart (either side of the date line) take the short way round, with
// the difference's own rounding error (Knuth's two-sum) kept, since what is left may be small.
// The half angle's sine has a condition number below 1 only up to half a turn: what is still
// beyond it (angles outside a turn) goes to float64.
constexpr float kHalfTurn = 3.1417f;  // pi (1 + 2^-15)
__device__ __forceinline__ float longitude_gap(const float4& a, const float4& b) {
  float d = __fsub_rn(a.y, b.y), low = __fsub_rn(a.w, b.w);
  if (fabsf(d) > 3.14159274f) {
    const float v = __fsub_rn(d, a.y);
    const float err = __fsub_rn(__fsub_rn(a.y, __fsub_rn(d, v)), __fadd_rn(b.y, v));
    const float turn = copysignf(6.28318548f, d);
    low = __fadd_rn(low, __fadd_rn(err, copysignf(1.74845553e-07f, d)));  // float(2 pi) is above 2 pi by this
    d = __fsub_rn(d, turn);
  }
  return __fadd_rn(d, low);
}

// One deferred entry of a small instance: the pair (i, j), i <= j, of type t goes to both
// of its places in the shared-memory matrix.
__device__ __forceinline__ void resolve_small(const MParams& P, const double* c, const double* cos64, int32_t* o,
                                              int L, int e, int& bad) {
  const int i = e >> 12, j = (e >> 1) & 2047, t = e & 1;
  const int32_t v = checked(minutes64(P, c, cos64, i, j, t), bad);
  o[t * L * L + i * L + j] = v;
  o[t * L * L + j * L + i] = v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Queue the lanes whose entry of type t is not certain in the CTA's queue (warp-uniform
// call); an entry past the queue's capacity is computed here.
__device__ __forceinline__ void enqueue(bool mine, int i, int j, int t, int* cq, unsigned& s_qn, int lane,
                                        const MParams& P, const double* c, const double* cos64, int32_t* o, int L,
                                        int& bad) {
  const unsigned m = __ballot_sync(0xffffffffu, mine);
  if (!m) return;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == leader) base = atomicAdd(&s_qn, static_cast<unsigned>(__popc(m)));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (!mine) return;
  const unsigned pos = base + __popc(m & ((1u << lane) - 1u));
  const int e = (i << 12) | (j << 1) | t;
  if (pos < kSmallQueue)
    cq[pos] = e;
  else
    resolve_small(P, c, cos64, o, L, e, bad);
}

// Small instances, each built whole in shared memory and written out by one bulk copy.
// The instance's scalars (S and the queue's length) alternate between two slots, so that
// thread 0 can clear the next instance's while this one's are read. Every evaluated pair
// stores its float32 results; the float64 drain after the queue barrier overwrites the
// uncertain ones. NT: the number of vehicle types.
template <bool HAV, int NT>
__global__ void __launch_bounds__(kSmallThreads, 8) travel_small_kernel(const __grid_constant__ MParams P) {
  __shared__ __align__(16) SmallStage st;
  __shared__ int cq[kSmallQueue];
  __shared__ unsigned s_mag[2], s_qn[2];
  const int lane = threadIdx.x & 31;
  const int nt = NT;
  const float k0 = P.k32[0], k1 = P.k32[1];
  const float two_r32 = static_cast<float>(P.two_r);
  int bad = 0;
  if (threadIdx.x < 2) s_mag[threadIdx.x] = s_qn[threadIdx.x] = 0u;
  __syncthreads();
  int par = 0;
  for (int b = blockIdx.x; b < P.B; b += gridDim.x) {
    const int lo = P.loc_off[b];
    const int L = P.loc_off[b + 1] - lo;
    if (!is_small(L, nt)) continue;
    const double* c = P.coords + 2 * static_cast<int64_t>(lo);
    int32_t* dst = P.travel + P.travel_off[b];
    // Every thread is past the previous instance's last barrier: its reads of the stage and
    // of its slots are done.
    if (threadIdx.x == 0) s_mag[par ^ 1] = s_qn[par ^ 1] = 0u;
    {
      const int l = threadIdx.x;  // L <= kSmallLoc <= kSmallThreads
      unsigned m = 0u;
      if (l < L) {
        double x = c[2 * l], y = c[2 * l + 1];
        if (HAV) {
          x *= P.deg;
          y *= P.deg;
        }
        const float xh = static_cast<float>(x), yh = static_cast<float>(y);
        if (HAV) {
          const double cx = cos(x);
          st.cos64[l] = cx;
          st.cphi[l] = static_cast<float>(cx);
          st.hl[l] = make_float4(xh, yh, static_cast<float>(x - static_cast<double>(xh)),
                                 static_cast<float>(y - static_cast<double>(yh)));
        } else {
          st.hl[l] = make_float4(xh, yh, 0.0f, 0.0f);
          m = __float_as_uint(fabsf(xh) + fabsf(yh));  // NaN's bits exceed every finite value
        }
      }
      if (!HAV) {
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0 && m) atomicMax(&s_mag[par], m);
      }
    }
    if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the last copy has read out
    __syncthreads();
    const int phase = static_cast<int>((reinterpret_cast<uintptr_t>(dst) >> 2) & 3u);
    int32_t* o = st.out + phase;  // o[w] is dst[w]; both 16-byte aligned at the same w
    const int LL = L * L;
    float c0, c1;  // the absolute part of each type's tolerance
    float rel = P.rel_hav;
    if (!HAV) {
      const float S = __uint_as_float(s_mag[par]);
      const float magk = 9.536743e-7f * S;  // 2^-20 S
      c0 = k0 * magk + 1e-6f;
      c1 = k1 * magk + 1e-6f;
      // every time is below 2 S k (1 + 10 2^-24); false for a NaN or infinite S
      rel = 2.0f * S * fmaxf(k0, NT > 1 ? k1 : 0.0f) * 1.001f < 4194304.0f ? 2e-6f : __int_as_float(0x7f800000);
    }
    // Pair p = f (L + 1) + k: row f from column f (k < L - f), else row L - 1 - f from column k - 1.
    const int L1 = L + 1, E = L * L1 / 2;
    int f = threadIdx.x / L1, k = threadIdx.x - f * L1;
    const int df = kSmallThreads / L1, dk = kSmallThreads - df * L1;
    for (int p0 = 0; p0 < E; p0 += kSmallThreads) {
      const bool live = p0 + static_cast<int>(threadIdx.x) < E;
      int i = f, j = f + k;
      if (k >= L - f) {
        i = L - 1 - f;
        j = k - 1;
      }
      if (!live) i = j = 0;
      f += df;
      k += dk;
      if (k >= L1) {
        k -= L1;
        ++f;
      }
      const float4 a = st.hl[i], bb = st.hl[j];
      float d32;
      bool screen = true;
      if (HAV) {
        const float dx = __fadd_rn(__fsub_rn(a.x, bb.x), __fsub_rn(a.z, bb.z));
        const float dy = longitude_gap(a, bb);
        const float s1 = sinf(__fmul_rn(dx, 0.5f)), s2 = sinf(__fmul_rn(dy, 0.5f));
        const float h = __fadd_rn(__fmul_rn(s1, s1), __fmul_rn(__fmul_rn(st.cphi[i], st.cphi[j]), __fmul_rn(s2, s2)));
        const float r = __fsqrt_rn(h);
        screen = r <= 0.9f && fmaxf(fabsf(dx), fabsf(dy)) <= kHalfTurn;
        d32 = __fmul_rn(two_r32, asinf(r));
        const float magk = two_r32 * 9.094947e-13f *  // 2 r 2^-40 (sum of |angles|)
                           (fabsf(a.x) + fabsf(bb.x) + fabsf(a.y) + fabsf(bb.y));
        c0 = k0 * magk + 1e-5f;
        c1 = k1 * magk + 1e-5f;
      } else {
        const float dx = __fsub_rn(a.x, bb.x), dy = __fsub_rn(a.y, bb.y);
        const float q = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
        d32 = q > 0.0f ? __fmul_rn(q, rsqrtf(q)) : q;  // sqrt(0) = 0 exactly; NaN stays NaN
      }
      if (!live) d32 = 0.0f;  // so that its stores write the 0 of entry (0, 0), whatever the coordinates
      int32_t v0, v1 = 0;
      const bool sure0 = round_screened_bounded(__fmul_rn(d32, k0), rel, c0, v0) && screen;
      const bool sure1 = NT < 2 || (round_screened_bounded(__fmul_rn(d32, k1), rel, c1, v1) && screen);
      o[i * L + j] = v0;
      o[j * L + i] = v0;
      if (NT > 1) {
        o[LL + i * L + j] = v1;
        o[LL + j * L + i] = v1;
      }
      if (__ballot_sync(0xffffffffu, live && !(sure0 && sure1))) {  // rare: float64 for these
        enqueue(live && !sure0, i, j, 0, cq, s_qn[par], lane, P, c, st.cos64, o, L, bad);
        if (NT > 1) enqueue(live && !sure1, i, j, 1, cq, s_qn[par], lane, P, c, st.cos64, o, L, bad);
      }
    }
    __syncthreads();  // the queue is complete
    const int nq = min(static_cast<int>(s_qn[par]), kSmallQueue);
    for (int e = threadIdx.x; e < nq; e += kSmallThreads) resolve_small(P, c, st.cos64, o, L, cq[e], bad);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the writes above, before the bulk copy reads them
    __syncthreads();
    const int W = nt * LL;
    const int head = min((4 - phase) & 3, W);
    const int mid = (W - head) & ~3;
    if (threadIdx.x == 0 && mid > 0) {
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + head),
                   "r"(smem_addr(o + head)), "r"(static_cast<uint32_t>(mid) * 4u)
                   : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    if (threadIdx.x < head) dst[threadIdx.x] = o[threadIdx.x];
    const int w = head + mid + static_cast<int>(threadIdx.x);
    if (w < W) dst[w] = o[w];
    par ^= 1;
  }
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // the last bulk copy is complete
  if (bad && P.status) atomicExch(P.status, ASCHED_E_INVALID);
}

// ------------------------------------------------------------------ tiles

// Tiles of an instance: the pairs I <= J of blocks of kTile locations.
__host__ __device__ __forceinline__ int64_t tiles_of(int L, int nt, bool skip_small) {
  const int64_t n = (static_cast<int64_t>(L) + kTile - 1) / kTile;
  return skip_small && is_small(L, nt) ? 0 : n * (n + 1) / 2;
}

// sin(x) for |x| <= pi / 2 (1 + 2^-12): x (1 + x^2 q(x^2)), q fitted for least relative error
// (6.1e-9) by Lawson's reweighted least squares. Its float32 value is within 3.6 * 2^-24.
__device__ __forceinline__ float sin_half(float x) {
  const float z = __fmul_rn(x, x);
  float q = __fmaf_rn(2.605750296424958e-06f, z, -1.980959059437737e-04f);
  q = __fmaf_rn(q, z, 8.33306647837162e-03f);
  q = __fmaf_rn(q, z, -1.6666659712791443e-01f);
  return __fmaf_rn(__fmul_rn(x, z), q, x);
}

// asin(sqrt(h)) for 0 <= h <= 1 / 4: r (1 + h q(h)) with r = sqrt(h), q as above (4.9e-9).
__device__ __forceinline__ float asin_root(float r, float h) {
  float q = __fmaf_rn(4.216628521680832e-02f, h, 2.4179525673389435e-02f);
  q = __fmaf_rn(q, h, 4.547037556767464e-02f);
  q = __fmaf_rn(q, h, 7.495297491550446e-02f);
  q = __fmaf_rn(q, h, 1.6666752099990845e-01f);
  return __fmaf_rn(__fmul_rn(r, h), q, r);
}

struct Deferred {  // an entry left to float64: pair (i, j) of instance b, type t
  int b, i, j, t;
};

__device__ __forceinline__ int32_t deferred_value(const MParams& P, const Deferred& e, int& bad) {
  const double* c = P.coords + 2 * static_cast<int64_t>(P.loc_off[e.b]);
  return checked(minutes64(P, c, nullptr, e.i, e.j, e.t), bad);
}

// Instances by tiles of 64 x 64 location pairs, every unordered pair evaluated once: the
// row block's entries go straight to global memory, the mirrored ones through shared
// memory, so that both leave by rows. Each CTA takes an equal run of consecutive tiles of
// all instances together (`tiles` of them), which it finds by a prefix sum over the
// instances; entries that float32 leaves open wait in a queue over the CTA's whole run, so
// that float64 works on full warps. Bound by float32 issue (about 60 instructions a
// Haversine pair) and by the float64 of the open entries. With one CTA per instance the
// largest instance's CTA set the time: 96 Haversine instances of 40 to 1,000 locations
// 2,364 us; by tiles, without library sines and arcsines and without float64 cosines per
// location, 56 us (60 MB written).
template <bool HAV, int NT>
__global__ void __launch_bounds__(kThreads, 4) travel_tiles_kernel(const __grid_constant__ MParams P, bool skip_small,
                                                                   int64_t tiles) {
  __shared__ float4 hl[2 * kTile];  // (x hi, y hi, x lo, y lo) of the row block, then of the column block
  __shared__ float cphi[2 * kTile];
  __shared__ int32_t mirror[NT][kTile][kTile + 1];
  __shared__ Deferred queue[kTileQueue];
  __shared__ unsigned s_mag[2], s_qn;
  __shared__ int s_b;
  __shared__ int64_t s_sum[kWarps], s_at;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float k0 = P.k32[0], k1 = P.k32[1];
  const float two_r32 = static_cast<float>(P.two_r);
  int64_t t0 = tiles * blockIdx.x / gridDim.x;
  const int64_t t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  int bad = 0;
  {  // the instance that holds tile t0: every thread sums a run of instances, then a prefix over threads
    const int per = (P.B + kThreads - 1) / kThreads;
    const int b0 = min(tid * per, P.B), b1 = min(b0 + per, P.B);
    int64_t mine = 0;
    for (int b = b0; b < b1; ++b) mine += tiles_of(P.loc_off[b + 1] - P.loc_off[b], NT, skip_small);
    int64_t upto = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    if (lane == 31) s_sum[warp] = upto;
    if (tid < 2) s_mag[tid] = 0u;
    if (tid == 0) s_qn = 0u;
    __syncthreads();
    for (int w = 0; w < warp; ++w) upto += s_sum[w];
    int64_t at = upto - mine;
    if (t0 < t1 && at <= t0 && t0 < upto) {  // one thread
      int b = b0;
      while (true) {
        const int64_t n = tiles_of(P.loc_off[b + 1] - P.loc_off[b], NT, skip_small);
        if (t0 < at + n) break;
        at += n;
        ++b;
      }
      s_b = b;
      s_at = at;
    }
    __syncthreads();
  }
  if (t0 >= t1) return;
  int b = s_b, par = 0;
  int64_t at = s_at;  // tiles before instance b
  for (int64_t t = t0; t < t1; ++t, par ^= 1) {
    int lo = P.loc_off[b], L = P.loc_off[b + 1] - lo;
    int64_t n = tiles_of(L, NT, skip_small);
    while (t >= at + n) {
      at += n;
      ++b;
      lo = P.loc_off[b];
      L = P.loc_off[b + 1] - lo;
      n = tiles_of(L, NT, skip_small);
    }
    const double* c = P.coords + 2 * static_cast<int64_t>(lo);
    int32_t* const base = P.travel + P.travel_off[b];
    const int64_t LL = static_cast<int64_t>(L) * L;
    // tile q is (I, J) with q = J (J + 1) / 2 + I
    const int64_t q = t - at;
    int J = static_cast<int>((sqrt(static_cast<float>(8 * q + 1)) - 1.0f) * 0.5f);
    while (static_cast<int64_t>(J) * (J + 1) / 2 > q) --J;
    while (static_cast<int64_t>(J + 1) * (J + 2) / 2 <= q) ++J;
    const int I = static_cast<int>(q - static_cast<int64_t>(J) * (J + 1) / 2);
    const int i0 = I * kTile, j0 = J * kTile;
    if (tid < 2 * kTile) {  // locations past the end repeat the last one; their entries are not written
      const int l = min((tid < kTile ? i0 : j0 - kTile) + tid, L - 1);
      double x = c[2 * l], y = c[2 * l + 1];
      if (HAV) {
        x = __dmul_rn(x, P.deg);
        y = __dmul_rn(y, P.deg);
      }
      const float xh = static_cast<float>(x), yh = static_cast<float>(y);
      float xl = 0.0f, yl = 0.0f;
      if (HAV) {
        xl = static_cast<float>(x - static_cast<double>(xh));
        yl = static_cast<float>(y - static_cast<double>(yh));
        cphi[tid] = __fmaf_rn(-xl, sinf(xh), cosf(xh));
      }
      hl[tid] = make_float4(xh, yh, xl, yl);
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(xh) + fabsf(yh)));  // a NaN's bits are largest
      if (lane == 0) atomicMax(&s_mag[par], m);
    }
    if (tid == 0) s_mag[par ^ 1] = 0u;
    __syncthreads();
    const float S = __uint_as_float(s_mag[par]);  // the largest |x| + |y| of the tile's locations
    float c0, c1, rel;
    if (HAV) {
      const float magk = two_r32 * 9.094947e-13f * 2.0f * S;  // 2 r 2^-40 (sum of |angles|)
      c0 = __fmaf_rn(k0, magk, 1e-5f);
      c1 = __fmaf_rn(k1, magk, 1e-5f);
      rel = P.rel_hav * 0.5f;
    } else {
      const float magk = 9.536743e-7f * S;  // 2^-20 S
      c0 = __fmaf_rn(k0, magk, 1e-6f);
      c1 = __fmaf_rn(k1, magk, 1e-6f);
      // every time is below 2 S k (1 + 10 2^-24); false for a NaN or infinite S
      rel = 2.0f * S * fmaxf(k0, NT > 1 ? k1 : 0.0f) * 1.001f < 4194304.0f ? 2e-6f : __int_as_float(0x7f800000);
    }
    const bool diagonal = I == J;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int jl = lane + 32 * h, j = j0 + jl;
      if (j0 + 32 * h >= L) break;
      const bool live = j < L;
      const float4 bb = hl[kTile + jl];
      const float cj = HAV ? cphi[kTile + jl] : 0.0f;
      const int rows = min(kTile, L - i0);
      int32_t* out = base + static_cast<int64_t>(i0 + warp) * L + j;
      for (int il = warp; il < rows; il += kWarps, out += static_cast<int64_t>(kWarps) * L) {
        const float4 a = hl[il];
        float d32;
        bool screen = true;
        if (HAV) {
          const float dx = __fadd_rn(__fsub_rn(a.x, bb.x), __fsub_rn(a.z, bb.z));
          const float dy = longitude_gap(a, bb);
          const float s1 = sin_half(__fmul_rn(dx, 0.5f)), s2 = sin_half(__fmul_rn(dy, 0.5f));
          const float g = __fmaf_rn(__fmul_rn(cphi[il], cj), __fmul_rn(s2, s2), __fmul_rn(s1, s1));
          const float r = g > 0.0f ? __fmul_rn(g, rsqrtf(g)) : g;  // sqrt(0) = 0 exactly; NaN stays NaN
          float angle = asin_root(r, g);
          screen = r <= 0.9f && fmaxf(fabsf(dx), fabsf(dy)) <= kHalfTurn;  // else the fits do not hold
          if (g > 0.25f) angle = asinf(r);
          d32 = __fmul_rn(two_r32, angle);
        } else {
          const float dx = __fsub_rn(a.x, bb.x), dy = __fsub_rn(a.y, bb.y);
          const float g = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
          d32 = g > 0.0f ? __fmul_rn(g, rsqrtf(g)) : g;
        }
        int32_t v0, v1 = 0;
        const bool sure0 = round_screened_bounded(__fmul_rn(d32, k0), rel, c0, v0) && screen;
        const bool sure1 = NT < 2 || (round_screened_bounded(__fmul_rn(d32, k1), rel, c1, v1) && screen);
        if (live && !(sure0 && sure1)) {  // rare: float64, later if the queue has room
#pragma unroll
          for (int ty = 0; ty < NT; ++ty) {
            if (ty == 0 ? sure0 : sure1) continue;
            const Deferred e{b, i0 + il, j, ty};
            const unsigned pos = atomicAdd(&s_qn, 1u);
            if (pos < kTileQueue) {
              queue[pos] = e;
            } else {
              const int32_t v = deferred_value(P, e, bad);
              if (ty == 0) v0 = v;
              else v1 = v;
            }
          }
        }
        if (live) {
          out[0] = v0;
          if (NT > 1) out[LL] = v1;
        }
        if (!diagonal) {
          mirror[0][jl][il] = v0;
          if (NT > 1) mirror[NT - 1][jl][il] = v1;
        }
      }
    }
    __syncthreads();
    const unsigned waiting = s_qn;  // nothing queues before the next tile's first barrier
    if (!diagonal) {
      const int cols = min(kTile, L - j0);  // the row block is full: I < J
      for (int jl = warp; jl < cols; jl += kWarps) {
        int32_t* out = base + static_cast<int64_t>(j0 + jl) * L + i0 + lane;
#pragma unroll
        for (int ty = 0; ty < NT; ++ty) {
          out[ty * LL] = mirror[ty][jl][lane];
          out[ty * LL + 32] = mirror[ty][jl][lane + 32];
        }
      }
    }
    if (waiting >= kTileQueue / 2 || t + 1 == t1) {  // uniform over the block
      __syncthreads();  // the float32 values of the entries are written
      const int nq = min(static_cast<int>(waiting), kTileQueue);
      for (int k = tid; k < nq; k += kThreads) {
        const Deferred e = queue[k];
        const int32_t v = deferred_value(P, e, bad);
        const int eL = P.loc_off[e.b + 1] - P.loc_off[e.b];
        int32_t* o = P.travel + P.travel_off[e.b] + static_cast<int64_t>(e.t) * eL * eL;
        o[static_cast<int64_t>(e.i) * eL + e.j] = v;
        o[static_cast<int64_t>(e.j) * eL + e.i] = v;
      }
      __syncthreads();
      if (tid == 0) s_qn = 0u;
    }
  }
  if (bad && P.status) atomicExch(P.status, ASCHED_E_INVALID);
}

}  // namespace

extern "C" int asched_travel_matrix(const asched_travel_spec* spec, int32_t* travel, int32_t* status,
                                    void* stream) {
  const asched_nvtx::Range nvtx_range("asched_travel_matrix");
  if (!spec || !travel) return ASCHED_E_INVALID;
  const int B = spec->n_instances;
  if (B < 0 || spec->n_types < 1 || spec->n_types > 2) return ASCHED_E_INVALID;
  if (spec->metric != ASCHED_METRIC_EUCLIDEAN && spec->metric != ASCHED_METRIC_HAVERSINE) return ASCHED_E_INVALID;
  for (int t = 0; t < spec->n_types; ++t)
    if (!(spec->speed_kmh[t] > 0.0) || !isfinite(spec->speed_kmh[t])) return ASCHED_E_INVALID;
  if (spec->metric == ASCHED_METRIC_HAVERSINE && !(spec->radius_km >= 0.0 && isfinite(spec->radius_km)))
    return ASCHED_E_INVALID;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (status && cudaMemsetAsync(status, 0, sizeof(int32_t), st) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  if (B == 0) return ASCHED_OK;
  if (!spec->h_loc_off || !spec->loc_off || !spec->travel_off || !spec->coords) return ASCHED_E_INVALID;
  if (spec->h_loc_off[0] != 0) return ASCHED_E_INVALID;
  for (int b = 0; b < B; ++b)
    if (spec->h_loc_off[b + 1] - spec->h_loc_off[b] < 1) return ASCHED_E_INVALID;
  MParams q = {};
  q.B = B;
  q.nt = spec->n_types;
  q.metric = spec->metric;
  q.speed[0] = spec->speed_kmh[0];
  q.speed[1] = spec->n_types > 1 ? spec->speed_kmh[1] : 1.0;
  q.k32[0] = static_cast<float>(60.0 / q.speed[0]);
  q.k32[1] = static_cast<float>(60.0 / q.speed[1]);
  const double r = spec->radius_km > 0.0 ? spec->radius_km : 6371.0;
  q.two_r = 2.0 * r;
  {  // every Haversine time is at most pi r 60 / speed (a float32 margin of 2^-10)
    const double kmax = 60.0 / (q.nt > 1 && q.speed[1] < q.speed[0] ? q.speed[1] : q.speed[0]);
    q.rel_hav = 3.141592653589793 * r * kmax * (1.0 + 1.0 / 1024.0) < 4194304.0 ? 8e-6f : INFINITY;
  }
  q.deg = 3.141592653589793 / 180.0;
  q.loc_off = spec->loc_off;
  q.travel_off = spec->travel_off;
  q.coords = spec->coords;
  q.travel = travel;
  q.status = status;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  int64_t n_small = 0;
  for (int b = 0; b < B; ++b) n_small += is_small(spec->h_loc_off[b + 1] - spec->h_loc_off[b], q.nt);
  const bool hav = q.metric == ASCHED_METRIC_HAVERSINE;
  // Small instances take their own kernel where they are all the batch holds or fill the chip
  // (4 per SM); a few among larger ones join the tiles, which saves a launch and its tail. Per
  // call, own kernel against tiles: 300 instances of 20 locations 8.4 against 10.4 us, of 52 with
  // two types 10.5 against 12.5, of 78 12.5 against 16.6 (Haversine 20.8 against 27.9). An
  // instance wider than a tile is three tiles, so where there is no more than one per SM the
  // tiles spread it better: 64 of 78 locations 12.5 against 12.0, Haversine 19.5 against 17.7.
  bool skip_small = n_small >= static_cast<int64_t>(sms) * 4;
  if (!skip_small && n_small == B) {
    int widest = 0;
    for (int b = 0; b < B; ++b) {
      const int L = spec->h_loc_off[b + 1] - spec->h_loc_off[b];
      widest = L > widest ? L : widest;
    }
    skip_small = widest <= kTile || n_small > sms;
  }
  int64_t tiles = 0;
  if (!skip_small || n_small < B)
    for (int b = 0; b < B; ++b) tiles += tiles_of(spec->h_loc_off[b + 1] - spec->h_loc_off[b], q.nt, skip_small);
  if (skip_small) {
    void (*const kernels[2][2])(MParams) = {{travel_small_kernel<false, 1>, travel_small_kernel<false, 2>},
                                            {travel_small_kernel<true, 1>, travel_small_kernel<true, 2>}};
    void (*const kern)(MParams) = kernels[hav][q.nt - 1];
    // eight 28 KB CTAs per SM want the largest shared-memory carveout (a per-device
    // attribute of the function, so it is set on every call: a host call, no device work)
    if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
        cudaSuccess) {
      (void)cudaGetLastError();
      return ASCHED_E_CUDA;
    }
    const int64_t cap = static_cast<int64_t>(sms) * 8;  // 8 CTAs of 128 threads per SM
    const int grid = static_cast<int>(n_small < cap ? n_small : cap);
    kern<<<grid, kSmallThreads, 0, st>>>(q);
    if (cudaGetLastError() != cudaSuccess) return ASCHED_E_CUDA;
  }
  if (tiles > 0) {
    void (*const kernels[2][2])(MParams, bool, int64_t) = {{travel_tiles_kernel<false, 1>, travel_tiles_kernel<false, 2>},
                                                           {travel_tiles_kernel<true, 1>, travel_tiles_kernel<true, 2>}};
    const int64_t cap = static_cast<int64_t>(sms) * 4;  // 4 CTAs of 256 threads per SM
    const int grid = static_cast<int>(tiles < cap ? tiles : cap);
    kernels[hav][q.nt - 1]<<<grid, kThreads, 0, st>>>(q, skip_small, tiles);
    if (cudaGetLastError() != cudaSuccess) return ASCHED_E_CUDA;
  }
  return ASCHED_OK;
}
