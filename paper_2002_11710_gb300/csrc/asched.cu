// asched.cu - host side of the searches: the C ABI of include/asched.h, launch shapes and
// launches. The device code is in search.cuh (one instance, full evaluation), carry.cuh (the
// same search with move values carried between iterations), batch.cu and serving.cu.
#include "kernels.h"
#include "nvtx_range.h"

#include <math.h>

namespace {

// ------------------------------------------------------------------ host side ------

// Shared-memory layout for an instance: the gather tables when they fit, else the
// int16 matrix (whose stamps limit iterations + tenure to 32,767). What a call accepts
// follows from it for every search, also those that then carry move values. rp: the batch and
// serving kernels' layout, with the RP records.
int choose_layout(int M, int V, int L, int nt, const asched_params* p, int limit_bytes, bool rp, Layout* out) {
  const Layout small = make_layout(M, V, L, nt, false, rp);
  if (!(p->flags & ASCHED_COMPACT_LAYOUT) && static_cast<int64_t>(small.total) * 4 + 64 <= limit_bytes) {
    *out = small;
    return ASCHED_OK;
  }
  const Layout big = make_layout(M, V, L, nt, true, rp);
  if (static_cast<int64_t>(big.total) * 4 + 64 > limit_bytes) return ASCHED_E_TOO_LARGE;
  if (static_cast<int64_t>(p->iterations) + p->tenure > 32767) return ASCHED_E_TOO_LARGE;
  *out = big;
  return ASCHED_OK;
}

int check_sizes(const asched_instance* inst, const asched_params* p) {
  if (!inst || !p) return ASCHED_E_INVALID;
  if (inst->n_loc < 1 || inst->n_types < 1 || inst->n_types > 2) return ASCHED_E_INVALID;
  if (inst->n_vehicles < 1 || inst->n_missions < 0) return ASCHED_E_INVALID;
  if (inst->n_vehicles > kMaxVehicles || inst->n_missions > kMaxMissions ||
      inst->n_missions + inst->n_vehicles > kMaxNodes)
    return ASCHED_E_TOO_LARGE;
  if (inst->duty_cap < 0 || inst->horizon < 0) return ASCHED_E_INVALID;
  if (p->tenure < 0 || p->iterations < 0 || p->lambda < 0) return ASCHED_E_INVALID;
  if (p->cap_mode != ASCHED_HARD && p->cap_mode != ASCHED_PENALTY) return ASCHED_E_INVALID;
  if (p->cluster_size != 0 && p->cluster_size != 1 && p->cluster_size != 2 && p->cluster_size != 4 &&
      p->cluster_size != 8 && p->cluster_size != 16)
    return ASCHED_E_INVALID;
  if (p->block_threads != 0 && (p->block_threads < 64 || p->block_threads > kMaxThreads || p->block_threads % 32))
    return ASCHED_E_INVALID;
  if (p->timeout_ns < 0 || (p->flags & ~(ASCHED_COMPACT_LAYOUT | ASCHED_TEST_WITHHOLD_KEY | ASCHED_PLAIN_LAUNCH)) != 0)
    return ASCHED_E_INVALID;
  if (p->grid_clusters < 0 || p->grid_clusters > kMaxGridClusters) return ASCHED_E_INVALID;
  return ASCHED_OK;
}


int max_smem_optin() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return -1;
  return v;
}

// Clusters of C CTAs (threads each, smem bytes of shared memory) that the device can
// hold at once for kernel fn; 0 when none fits.
int active_clusters(void* fn, int C, int threads, int smem, int* out) {
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return ASCHED_E_CUDA;
  if (C > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return ASCHED_E_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(smem);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  *out = n;
  return ASCHED_OK;
}

// Warps per CTA for a neighbourhood of `chunks` 32-item chunks dealt over `ctas` CTAs:
// the fewest, in steps of 4 (equal shares for an SM's four schedulers), that keep the
// largest per-warp share at its least (16 warps at most).
int warps_for(int64_t chunks, int64_t ctas) {
  const int64_t least = (chunks + 16 * ctas - 1) / (16 * ctas);
  int w = 4;
  while (w < 16 && (chunks + w * ctas - 1) / (w * ctas) > least) w += 4;
  return w;
}

// Bytes of the global key slots a launch of K clusters uses: two buffers of K keys,
// each buffer in its own 128-byte lines.
int64_t grid_slot_stride(int K) { return round_up(K, 16); }  // in uint64 words
size_t grid_workspace_bytes(int K) { return K > 1 ? static_cast<size_t>(2 * grid_slot_stride(K) * 8) : 0; }

// More than 4 chunks of 32 items (relocation pairs, then swaps) per warp of a full cluster.
bool wide_search(const asched_instance* inst) {
  const int64_t M = inst->n_missions, V = inst->n_vehicles;
  const int64_t evals = (M + V) * ((M + 1) / 2) + M * (M - 1) / 2;
  return (evals + 31) / 32 > 4 * 16 * static_cast<int64_t>(kMaxCluster);
}

// Launch shape (block size, cluster size C and clusters K) and the form of the search it runs
// (its kernel and layout); returns status.
// allow_grid: the call has a workspace for the keys between clusters (K may exceed 1).
int make_plan(const asched_instance* inst, const asched_params* p, bool debug, bool allow_grid,
              asched_plan_t* plan, Layout* lay_out, void** fn_out) {
  int rc = check_sizes(inst, p);
  if (rc != ASCHED_OK) return rc;
  if (p->grid_clusters < 0 || (!allow_grid && p->grid_clusters > 1)) return ASCHED_E_INVALID;
  const int M = inst->n_missions, V = inst->n_vehicles;
  const int limit = max_smem_optin();
  if (limit < 0) return ASCHED_E_CUDA;
  Layout lay;
  rc = choose_layout(M, V, inst->n_loc, inst->n_types, p, limit, false, &lay);
  if (rc != ASCHED_OK) return rc;
  const int bytes = lay.total * 4;
  void* fn = asched_kernels::full(p->cap_mode == ASCHED_PENALTY, inst->deadline != nullptr, debug, lay.big);
  const int64_t items = static_cast<int64_t>(M + V) * M + static_cast<int64_t>(M) * (M - 1) / 2;
  const int64_t evals = static_cast<int64_t>(M + V) * ((M + 1) / 2) + static_cast<int64_t>(M) * (M - 1) / 2;
  const int64_t chunks = (evals + 31) / 32;
  // Neighbourhoods of 1,024 items or more take the largest cluster. The evaluation deals
  // 32-item chunks of its item list (relocation pairs, then swaps) round-robin over the
  // warps of every CTA, so an iteration lasts as long as the warp with the most chunks,
  // plus a little per warp (reduce, decode, rewrite, barriers): such neighbourhoods take
  // the fewest warps per CTA that keep that largest share at its least (warps_for).
  // Measured on neighbourhoods of 1,778 to 259,800 moves, this was the fastest shape or
  // within 1 % of it. Smaller neighbourhoods take one thread per item and the fewest CTAs
  // that cover them.
  const bool wide = items >= 1024;
  int cl = p->cluster_size;
  if (cl == 0 && wide) cl = kMaxCluster;
  int K = p->grid_clusters > 0 ? p->grid_clusters : 1;
  const int probe_threads = p->block_threads ? p->block_threads : kMaxThreads;
  if (p->cluster_size == 0 && cl > 1) {
    // shrink the cluster until the device can place one
    int n = 0;
    while (cl > 1) {
      rc = active_clusters(fn, cl, probe_threads, bytes, &n);
      if (rc != ASCHED_OK) return rc;
      if (n > 0) break;
      cl /= 2;
    }
  }
  // Neighbourhoods with more than 4 chunks per warp on one full cluster (the evaluation
  // then dominates the iteration) spread over every cluster of that size the device
  // holds at once, when the call has a workspace. The largest cluster is kept: keys
  // cross clusters through L2, which costs about 2 us per iteration whatever the number
  // of clusters, so fewer, larger clusters (more of the exchange in DSMEM) measured
  // fastest (on the large instance 7 x 16 CTAs: 3.7 us per iteration; 15 x 8: 3.8;
  // 27 x 4: 4.1; 76 x 2: 5.2).
  if (allow_grid && p->grid_clusters == 0 && wide && wide_search(inst)) {
    int n = 0;
    rc = active_clusters(fn, cl, probe_threads, bytes, &n);
    if (rc != ASCHED_OK) return rc;
    if (n >= 2) K = n;
  }
  if (cl == 0) cl = 1;
  int threads = p->block_threads;
  if (threads == 0) {
    if (wide) {
      threads = 32 * warps_for(chunks, static_cast<int64_t>(cl) * K);
    } else {
      const int64_t want = items > M + V ? items : M + V;
      threads = want >= kMaxThreads ? kMaxThreads : (want <= 64 ? 64 : round_up(static_cast<int>(want), 32));
    }
  }
  if (p->cluster_size == 0 && !wide && K == 1) {
    cl = 1;
    while (cl < kMaxCluster && items > static_cast<int64_t>(cl) * threads) cl *= 2;
    int n = 0;
    while (cl > 1) {  // shrink the cluster until the device can place one
      rc = active_clusters(fn, cl, threads, bytes, &n);
      if (rc != ASCHED_OK) return rc;
      if (n > 0) break;
      cl /= 2;
    }
  }
  if (K > 1) {  // every cluster must be resident at once
    int n = 0;
    rc = active_clusters(fn, cl, threads, bytes, &n);
    if (rc != ASCHED_OK) return rc;
    if (K > n) return ASCHED_E_TOO_LARGE;
  }
  // Carried move values on one cluster only. Over several, an iteration's chain of table
  // updates comes on top of the exchange through L2, and the full evaluation's share per warp is
  // small: 7 x 16 CTAs, carried against full, 400 missions and 50 vehicles 8.5 against 6.7 us an
  // iteration, 800 and 20 16.1 against 11.3, 1,200 and 30 22.9 against 18.5.
  Layout form;
  const int kind = debug || K > 1 ? SEARCH_TABLES
                                  : pick_search(M, V, inst->n_loc, inst->n_types, inst->deadline != nullptr, cl,
                                                threads / 32, p->tenure, (p->flags & ASCHED_COMPACT_LAYOUT) != 0,
                                                lay.big, false, (limit - 64) / 4, &form);
  if (kind == SEARCH_CARRY32 || kind == SEARCH_CARRY16) {
    void* cfn = asched_kernels::carry(p->cap_mode == ASCHED_PENALTY, inst->deadline != nullptr, kind == SEARCH_CARRY16);
    int n = 1;
    if (cl > 1) {
      rc = active_clusters(cfn, cl, threads, form.total * 4, &n);
      if (rc != ASCHED_OK) return rc;
    }
    if (n > 0) {  // else the full evaluation, which is placed above
      fn = cfn;
      lay = form;
    }
  }
  plan->cluster_size = cl;
  plan->block_threads = threads;
  plan->smem_bytes = lay.total * 4;
  plan->moves_per_iteration = moves_of(M, V);
  plan->grid_clusters = K;
  plan->workspace_bytes = static_cast<int64_t>(grid_workspace_bytes(K));
  if (lay_out) *lay_out = lay;
  if (fn_out) *fn_out = fn;
  return ASCHED_OK;
}

int launch(const asched_instance* inst, const asched_params* p, bool debug, KParams kp, void* workspace,
           size_t ws_bytes, bool allow_grid, void* stream) {
  asched_plan_t plan;
  Layout lay;
  void* fn;
  int rc = make_plan(inst, p, debug, allow_grid, &plan, &lay, &fn);
  if (rc != ASCHED_OK) return rc;
  if (!inst->travel || !inst->veh_base) return ASCHED_E_INVALID;
  if (inst->n_missions > 0 && (!inst->pickup || !inst->delivery)) return ASCHED_E_INVALID;
  const int K = plan.grid_clusters;
  if (K > 1 && (!workspace || ws_bytes < grid_workspace_bytes(K) || (reinterpret_cast<uintptr_t>(workspace) & 127u)))
    return ASCHED_E_INVALID;
  const bool pen = p->cap_mode == ASCHED_PENALTY;
  kp.travel = inst->travel;
  kp.veh_base = inst->veh_base;
  kp.veh_type = inst->veh_type;
  kp.pickup = inst->pickup;
  kp.delivery = inst->delivery;
  kp.heli_only = inst->heli_only;
  kp.deadline = inst->deadline;
  kp.L = inst->n_loc;
  kp.nt = inst->n_types;
  kp.V = inst->n_vehicles;
  kp.M = inst->n_missions;
  kp.cap = inst->duty_cap;
  kp.horizon = inst->horizon;
  kp.tenure = p->tenure;
  kp.iterations = p->iterations;
  kp.lambda = pen ? p->lambda : 0;
  kp.cluster = plan.cluster_size;
  kp.grid_clusters = K;
  kp.gslot_stride = static_cast<int32_t>(grid_slot_stride(K));
  kp.gslots = K > 1 ? static_cast<uint64_t*>(workspace) : nullptr;
  kp.timeout_ns = p->timeout_ns > 0 ? p->timeout_ns : kDefaultTimeoutNs;
  kp.test_withhold = (p->flags & ASCHED_TEST_WITHHOLD_KEY) ? 1 : 0;
  kp.lay = lay;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.smem_bytes) != cudaSuccess)
    return ASCHED_E_CUDA;
  if (plan.cluster_size > 8 &&
      cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return ASCHED_E_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (K > 1 && cudaMemsetAsync(workspace, 0, grid_workspace_bytes(K), st) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.cluster_size * K, 1, 1);
  cfg.blockDim = dim3(plan.block_threads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(plan.smem_bytes);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.cluster_size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // Clusters that wait on one another need to be resident together: a cooperative
  // launch guarantees it (or fails to launch).
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = (K > 1 && !(p->flags & ASCHED_PLAIN_LAUNCH)) ? 2 : 1;
  void* args[] = {&kp};
  if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  return ASCHED_OK;
}

// One way to run a batch: CTAs of `threads`, per_sm of them on an SM at once.
struct BatchForm {
  int threads, per_sm;
  int limit_words;  // shared memory by which each instance's form is chosen
  int words;        // the most any of them takes
  int places;       // instances (CTAs or clusters) at once
  double time;      // estimate of an iteration of all
};

// The estimate, in items of the full evaluation (see carry_cost): an iteration of an instance takes
// 208 + c r / (C e(r W)) with r CTAs of W warps on its SM, e(w) = 24 w / (w + 8) the items an SM gets
// done with w warps (200 missions on 3 vehicles by the full evaluation: 64 threads 83 us, 128 42.4,
// 256 25.1, 512 18.4; 208 items are 1.4 us). The longest start first. A batch takes the longest,
// whose SM is its own once its neighbours are through, or the sum over all places, or, with more
// instances than places, those that have to share one. Over 48 batches of 100 to 1,024 instances,
// equal and mixed, mostly within 15 %, and the choice within 3 % of the better one.
int batch_form(const asched_batch* bt, const asched_params* p, int C, int sms, int table_words, BatchForm* f) {
  const bool dl = bt->deadline != nullptr, compact = (p->flags & ASCHED_COMPACT_LAYOUT) != 0;
  const int W = f->threads / 32, r = f->per_sm, B = bt->n_instances;
  const auto per_item = [&](int k) { return k * (k * W + 8.0) / (24.0 * k * W * C); };  // with k CTAs on the SM
  constexpr int kFixed = 208, kBins = 16 * 24;  // 16 per octave of an instance's items
  int bins[kBins] = {};
  double sum = 0.0, most = 0.0;
  f->words = 0;
  for (int b = 0; b < B; ++b) {
    const int L = bt->h_loc_off[b + 1] - bt->h_loc_off[b], V = bt->h_veh_off[b + 1] - bt->h_veh_off[b],
              M = bt->h_mis_off[b + 1] - bt->h_mis_off[b];
    const bool half = compact || make_layout(M, V, L, bt->n_types, false, true).total > table_words;
    Layout lay;
    const int kind = pick_search(M, V, L, bt->n_types, dl, C, W, p->tenure, compact, half, true, f->limit_words, &lay);
    if (lay.total > f->limit_words) return ASCHED_E_TOO_LARGE;
    if (lay.total > f->words) f->words = lay.total;
    const bool carried = kind == SEARCH_CARRY32 || kind == SEARCH_CARRY16;
    const double c = 1.0 + (carried ? 0.25 * carry_cost(M, V, dl, C, W) : static_cast<double>(search_items(M, V)));
    sum += c;
    most = c > most ? c : most;
    const int bin = static_cast<int>(16.0 * log2(c));
    ++bins[bin < kBins ? bin : kBins - 1];
  }
  const auto nth = [&](int n) {  // items of the n-th longest instance, n < B
    int bin = kBins - 1;
    for (int k = bins[bin]; k <= n; k += bins[bin]) --bin;
    return exp2((bin + 0.5) / 16.0);
  };
  f->places = sms * r / C;
  if (C > 1) {
    const int rc = active_clusters(asched_kernels::batch(p->cap_mode == ASCHED_PENALTY, dl, true), C, f->threads,
                                   f->words * 4, &f->places);
    if (rc != ASCHED_OK) return rc;
    if (f->places < 1) return ASCHED_E_TOO_LARGE;
  }
  const int sets = (f->places + r - 1) / r;  // SMs, or groups of C of them
  f->time = (kFixed * static_cast<double>(B) + sum * per_item(r)) / f->places;
  double longest = kFixed + most * per_item(1);
  if (B <= f->places && B > sets) longest += nth(sets) * (per_item(r) - per_item(1));
  for (int64_t j = 1; j * f->places < B; ++j) {  // of j places + 1 instances some place gets j + 1
    const int n = static_cast<int>(j) * f->places, rest = (B - n + sets - 1) / sets;
    const double all = (j + 1) * kFixed + nth(n) * (j * per_item(r) + per_item(rest < r ? rest : r));
    longest = all > longest ? all : longest;
  }
  f->time = longest > f->time ? longest : f->time;
  return ASCHED_OK;
}

int launch_batch(const asched_batch* bt, const asched_params* p, const asched_batch_result* out,
                 void* workspace, size_t ws_bytes, void* stream) {
  if (!bt || !p || !out) return ASCHED_E_INVALID;
  const int B = bt->n_instances;
  if (B < 0) return ASCHED_E_INVALID;
  if (B == 0) return ASCHED_OK;
  if (!bt->h_loc_off || !bt->h_veh_off || !bt->h_mis_off || !bt->loc_off || !bt->veh_off || !bt->mis_off ||
      !bt->travel_off || !bt->travel || !bt->veh_base || !bt->pickup || !bt->delivery || !bt->duty_cap ||
      !bt->horizon)
    return ASCHED_E_INVALID;
  if (!out->route_off || !out->route || !out->info || !workspace) return ASCHED_E_INVALID;
  if (ws_bytes < sizeof(int32_t) * (static_cast<size_t>(B) + 1)) return ASCHED_E_INVALID;
  const int limit = max_smem_optin();
  if (limit < 0) return ASCHED_E_CUDA;
  const int limit_words = (limit - 64) / 4;
  // CTAs per instance: 1 (one persistent CTA per SM slot) or a cluster of C CTAs
  const int C = p->cluster_size > 1 ? p->cluster_size : 1;
  asched_instance one = {};
  one.n_types = bt->n_types;
  one.duty_cap = 0;
  one.horizon = 0;
  for (int b = 0; b < B; ++b) {
    one.n_loc = bt->h_loc_off[b + 1] - bt->h_loc_off[b];
    one.n_vehicles = bt->h_veh_off[b + 1] - bt->h_veh_off[b];
    one.n_missions = bt->h_mis_off[b + 1] - bt->h_mis_off[b];
    int bad = check_sizes(&one, p);
    if (bad != ASCHED_OK) return bad;
    Layout lay;
    bad = choose_layout(one.n_missions, one.n_vehicles, one.n_loc, one.n_types, p, limit, true, &lay);
    if (bad != ASCHED_OK) return bad;
  }
  int dev = 0, sms = 0, sm_bytes = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  // The block: 512 threads one per SM, or, with more instances than that has places for, 256 threads
  // two per SM, by the estimate; a caller's block as many per SM as the estimate finds best. Two per
  // SM get more done (250 iterations of 304 instances, us each: 40 missions on 8 vehicles 3.1
  // against 4.4, 100 on 20 7.1 against 9.0, 200 on 30 13.2 against 15.4) and share 228 KB, where the
  // tables of a large instance with few vehicles do not fit and the carried form is slower (200 on
  // 3: 38.9 against 36.4); one finishes the longest instances of a mixed batch sooner (512 of 10 to
  // 200 missions on 3 to 30 vehicles 16.2 against 20.0, 1,024 of them 31.5 against 27.0).
  const int own = p->block_threads;
  BatchForm form = {own ? own : kMaxThreads, 1, limit_words, 0, 0, 0.0};
  int rc = batch_form(bt, p, C, sms, limit_words, &form);
  if (rc != ASCHED_OK) return rc;
  const int per_sm_most = own ? kMaxThreads / own : 2;
  for (int r = 2, places = form.places; r <= per_sm_most && B > places; r *= 2) {
    BatchForm f = {own ? own : kMaxThreads / r, r, (sm_bytes / r - 1024 - 64) / 4, 0, 0, 0.0};
    if (f.limit_words > limit_words) f.limit_words = limit_words;
    if (batch_form(bt, p, C, sms, limit_words, &f) != ASCHED_OK) break;
    places = f.places;
    if (f.time < form.time) form = f;
  }
  const int threads = form.threads;
  const int64_t bytes = static_cast<int64_t>(form.words) * 4;
  const bool pen = p->cap_mode == ASCHED_PENALTY;
  const bool dl = bt->deadline != nullptr;
  void* fn = asched_kernels::batch(pen, dl, C > 1);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes)) !=
      cudaSuccess)
    return ASCHED_E_CUDA;
  int grid = 0;
  if (C > 1) {
    int n = 0;
    rc = active_clusters(fn, C, threads, static_cast<int>(bytes), &n);
    if (rc != ASCHED_OK) return rc;
    if (n < 1) return ASCHED_E_TOO_LARGE;
    grid = (B < n ? B : n) * C;
  } else {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, static_cast<size_t>(bytes)) != cudaSuccess) {
      (void)cudaGetLastError();
      return ASCHED_E_CUDA;
    }
    if (per_sm < 1) return ASCHED_E_TOO_LARGE;
    grid = B < sms * per_sm ? B : sms * per_sm;
  }
  BParams q = {};
  q.run.nt = bt->n_types;
  q.run.tenure = p->tenure;
  q.run.iterations = p->iterations;
  q.run.lambda = pen ? p->lambda : 0;
  q.run.cluster = C;
  q.run.timeout_ns = p->timeout_ns > 0 ? p->timeout_ns : kDefaultTimeoutNs;
  q.B = B;
  q.table_words = limit_words;
  q.limit_words = form.limit_words;
  q.compact = (p->flags & ASCHED_COMPACT_LAYOUT) ? 1 : 0;
  q.loc_off = bt->loc_off;
  q.veh_off = bt->veh_off;
  q.mis_off = bt->mis_off;
  q.travel_off = bt->travel_off;
  q.travel = bt->travel;
  q.veh_base = bt->veh_base;
  q.veh_type = bt->veh_type;
  q.pickup = bt->pickup;
  q.delivery = bt->delivery;
  q.heli_only = bt->heli_only;
  q.deadline = bt->deadline;
  q.duty_cap = bt->duty_cap;
  q.horizon = bt->horizon;
  q.out_off = out->route_off;
  q.out_route = out->route;
  q.out_flight = out->flight;
  q.out_over = out->overflow;
  q.info = out->info;
  q.work = static_cast<int32_t*>(workspace);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  void* order_args[] = {const_cast<int32_t*>(&bt->n_instances), const_cast<const int32_t**>(&bt->veh_off),
                        const_cast<const int32_t**>(&bt->mis_off), &q.work};
  if (cudaLaunchKernel(asched_kernels::batch_order(), dim3((B + 255) / 256), dim3(256), order_args, 0, st) !=
      cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  void* args[] = {&q};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(bytes);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  return ASCHED_OK;
}

// Load every serving kernel now. Kernels are loaded on first use, and loading one can
// wait for the device to go idle: a second persistent launch started while a first one
// runs (the cluster lane and the one-CTA lane of a server) would then wait until the
// first ends, which for a persistent launch is only its idle timeout.
int preload_serve_kernels() {
  for (int k = 0; k < 8; ++k) {
    void* fn = asched_kernels::serve((k & 1) != 0, (k & 2) != 0, (k & 4) != 0);
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, fn) != cudaSuccess) {
      (void)cudaGetLastError();
      return ASCHED_E_CUDA;
    }
  }
  return ASCHED_OK;
}

int launch_serve(const asched_server* sv, const asched_params* p, int64_t idle_ns, int32_t max_ctas, void* stream) {
  if (!sv || !p) return ASCHED_E_INVALID;
  if (sv->n_slots < 1 || sv->ring_len < sv->n_slots || sv->max_loc < 1 || sv->max_vehicles < 1 ||
      sv->max_missions < 0 || sv->n_types < 1 || sv->n_types > 2 || idle_ns <= 0)
    return ASCHED_E_INVALID;
  if (!sv->slot_data || !sv->slot_out || !sv->ring || !sv->control || !sv->done) return ASCHED_E_INVALID;
  asched_instance cap = {};
  cap.n_loc = sv->max_loc;
  cap.n_types = sv->n_types;
  cap.n_vehicles = sv->max_vehicles;
  cap.n_missions = sv->max_missions;
  int rc = check_sizes(&cap, p);
  if (rc != ASCHED_OK) return rc;
  const int C = p->cluster_size > 1 ? p->cluster_size : 1;
  if (C > 1 && max_ctas > 0 && max_ctas < C) return ASCHED_E_INVALID;
  rc = preload_serve_kernels();
  if (rc != ASCHED_OK) return rc;
  const int limit = max_smem_optin();
  if (limit < 0) return ASCHED_E_CUDA;
  Layout lay;  // the largest request the slots can hold sizes the launch
  rc = choose_layout(sv->max_missions, sv->max_vehicles, sv->max_loc, sv->n_types, p, limit, true, &lay);
  if (rc != ASCHED_OK) return rc;
  const bool pen = p->cap_mode == ASCHED_PENALTY;
  const bool dl = sv->has_deadlines != 0;
  const int threads = p->block_threads ? p->block_threads : kMaxThreads;
  int dev = 0, sms = 0, sm_bytes = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  // Shared memory: the full evaluation of the largest request, or what carried values take at most
  // (every part of that layout grows with the sizes), but of the SM no more than the share that the
  // block's registers take, so that as many workers fit as threads allow, or another launch beside
  // workers of smaller blocks. With all of it, one worker an SM, by 128-thread workers: 2,048 requests
  // of 10 to 40 missions in slots for 40 5.4 ms against 2.2, 1,024 of 20 to 100 6.2 against 3.2.
  const int limit_words = (limit - 64) / 4;
  int words = lay.total;
  for (int t16 = 0; t16 < 2 && p->tenure <= kMaxCarryTenure; ++t16) {
    const int need = make_carry_layout(sv->max_missions, sv->max_vehicles, sv->max_loc, sv->n_types, dl, t16 != 0, true, C,
                                       threads / 32, p->tenure).total;
    words = need > words ? need : words;
  }
  const int64_t share = (static_cast<int64_t>(sm_bytes) * threads / kMaxThreads - 1024 - 64) / 4;
  if (words > share) words = static_cast<int>(share > lay.total ? share : lay.total);
  if (words > limit_words) words = limit_words;
  const int64_t bytes = static_cast<int64_t>(words) * 4;
  void* fn = asched_kernels::serve(pen, dl, C > 1);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes)) !=
      cudaSuccess)
    return ASCHED_E_CUDA;
  if (C > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return ASCHED_E_CUDA;
  SParams q = {};
  q.run.nt = sv->n_types;
  q.run.tenure = p->tenure;
  q.run.iterations = p->iterations;
  q.run.lambda = pen ? p->lambda : 0;
  q.run.cluster = C;
  q.run.timeout_ns = p->timeout_ns > 0 ? p->timeout_ns : kDefaultTimeoutNs;
  q.n_slots = sv->n_slots;
  q.ring_len = sv->ring_len;
  q.Lc = sv->max_loc;
  q.Vc = sv->max_vehicles;
  q.Mc = sv->max_missions;
  q.nt = sv->n_types;
  q.slot_words = serve_slot_words(q.Lc, q.Vc, q.Mc, q.nt);
  q.out_words = serve_out_words(q.Vc, q.Mc);
  q.limit_words = words;
  q.table_words = lay.total;
  q.compact = (p->flags & ASCHED_COMPACT_LAYOUT) ? 1 : 0;
  q.idle_ns = idle_ns;
  q.slot_data = sv->slot_data;
  q.slot_out = sv->slot_out;
  q.ring = sv->ring;
  q.control = sv->control;
  q.done = sv->done;
  void* args[] = {&q};
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(bytes);
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute attr[1];
  int grid;
  if (C > 1) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(C, 1, 1);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      return ASCHED_E_CUDA;
    }
    if (clusters < 1) return ASCHED_E_TOO_LARGE;
    int want = (max_ctas > 0 ? max_ctas : sms) / C;  // whole clusters only
    grid = C * (want < clusters ? want : clusters);
  } else {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, static_cast<size_t>(bytes)) !=
        cudaSuccess) {
      (void)cudaGetLastError();
      return ASCHED_E_CUDA;
    }
    if (per_sm < 1) return ASCHED_E_TOO_LARGE;
    grid = sms * per_sm;
    if (max_ctas > 0 && max_ctas < grid) grid = max_ctas;
  }
  cfg.gridDim = dim3(grid, 1, 1);
  if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  return ASCHED_OK;
}

}  // namespace

// ------------------------------------------------------------------ fixed scratch ---

// Work queue and processing order for asched_solve_batch_static: a fixed array in
// every device's global memory, so that call needs no workspace from its caller.
// Host code only uses its device address, looked up on each call (see below).
static __device__ __align__(256) int32_t g_batch_scratch[1 + ASCHED_STATIC_BATCH_MAX];

namespace {

// Device address of g_batch_scratch on the current device. Looked up on every call
// (the lookup allocates nothing), so the address stays right after a device reset,
// which reloads the module and may move the array. The first lookup on a device can
// load the module, so it belongs before any stream capture.
int static_scratch(void** out) {
  void* ptr = nullptr;
  if (cudaGetSymbolAddress(&ptr, g_batch_scratch) != cudaSuccess || !ptr) {
    (void)cudaGetLastError();
    return ASCHED_E_CUDA;
  }
  *out = ptr;
  return ASCHED_OK;
}

}  // namespace

// ------------------------------------------------------------------ C ABI ----------

extern "C" {

int asched_abi_version(void) { return ASCHED_ABI_VERSION; }

const char* asched_status_string(int status) {
  switch (status) {
    case ASCHED_OK: return "ok";
    case ASCHED_E_INVALID: return "invalid argument or instance data";
    case ASCHED_E_TOO_LARGE: return "instance too large for the on-chip layout";
    case ASCHED_E_OVERFLOW_GUARD: return "int32 objective could overflow";
    case ASCHED_E_INFEASIBLE_INIT: return "no feasible initial schedule";
    case ASCHED_E_TIMEOUT: return "a bounded device wait timed out";
    case ASCHED_E_CUDA: return "CUDA runtime error";
    default: return "unknown status";
  }
}

int asched_num_moves(int32_t n_missions, int32_t n_vehicles, int64_t* out) {
  if (!out || n_missions < 0 || n_vehicles < 1) return ASCHED_E_INVALID;
  *out = moves_of(n_missions, n_vehicles);
  return ASCHED_OK;
}

int asched_check_instance_host(const asched_instance* inst, const asched_params* p) {
  int rc = check_sizes(inst, p);
  if (rc != ASCHED_OK) return rc;
  const int L = inst->n_loc, V = inst->n_vehicles, M = inst->n_missions, nt = inst->n_types;
  if (!inst->travel || !inst->veh_base || (M > 0 && (!inst->pickup || !inst->delivery))) return ASCHED_E_INVALID;
  int64_t maxT = 0;
  for (int64_t i = 0; i < static_cast<int64_t>(nt) * L * L; ++i) {
    if (inst->travel[i] < 0) return ASCHED_E_INVALID;
    if (inst->travel[i] > maxT) maxT = inst->travel[i];
  }
  for (int v = 0; v < V; ++v) {
    if (inst->veh_base[v] < 0 || inst->veh_base[v] >= L) return ASCHED_E_INVALID;
    const int ty = inst->veh_type ? inst->veh_type[v] : 0;
    if (ty < 0 || ty >= nt) return ASCHED_E_INVALID;
  }
  for (int m = 0; m < M; ++m) {
    const int pk = inst->pickup[m], d = inst->delivery[m];
    if (pk < 0 || pk >= L || d < 0 || d >= L || pk == d) return ASCHED_E_INVALID;
    if (inst->heli_only && (inst->heli_only[m] < 0 || inst->heli_only[m] > 1)) return ASCHED_E_INVALID;
  }
  const double lam = p->cap_mode == ASCHED_PENALTY ? static_cast<double>(p->lambda) : 0.0;
  const double bound = 2.0 * (2.0 * M + V + 2.0) * static_cast<double>(maxT) * (1.0 + lam);
  if (!(bound < 2147483648.0)) return ASCHED_E_OVERFLOW_GUARD;
  return ASCHED_OK;
}

int asched_plan(const asched_instance* inst, const asched_params* params, asched_plan_t* out) {
  if (!out) return ASCHED_E_INVALID;
  return make_plan(inst, params, false, true, out, nullptr, nullptr);
}

namespace {
KParams solve_params(const int32_t* init_route_off, const int32_t* init_route, const asched_result* out) {
  KParams kp = {};
  kp.init_off = init_route_off;
  kp.init_route = init_route;
  kp.out_off = out->route_off;
  kp.out_route = out->route;
  kp.out_flight = out->flight;
  kp.out_over = out->overflow;
  kp.info = out->info;
  kp.traj_move = out->traj_move;
  kp.traj_z = out->traj_z;
  return kp;
}
}  // namespace

int asched_solve(const asched_instance* inst, const asched_params* params, const int32_t* init_route_off,
                 const int32_t* init_route, const asched_result* out, void* stream) {
  const asched_nvtx::Range nvtx_range("asched_solve");
  if (!out || !out->route_off || !out->route || !out->info) return ASCHED_E_INVALID;
  if ((init_route_off == nullptr) != (init_route == nullptr)) return ASCHED_E_INVALID;
  return launch(inst, params, false, solve_params(init_route_off, init_route, out), nullptr, 0, false, stream);
}

int asched_validate(const asched_instance* inst, const asched_params* params) {
  return asched_check_instance_host(inst, params);
}

int asched_workspace_bytes(const asched_instance* inst, const asched_params* params, size_t* bytes) {
  if (!bytes) return ASCHED_E_INVALID;
  asched_plan_t plan;
  const int rc = make_plan(inst, params, false, true, &plan, nullptr, nullptr);
  if (rc != ASCHED_OK) return rc;
  *bytes = static_cast<size_t>(plan.workspace_bytes);
  return ASCHED_OK;
}

int asched_greedy_init(const asched_instance* inst, const asched_params* params, int32_t* route_off,
                       int32_t* route, int32_t* info, void* stream) {
  const asched_nvtx::Range nvtx_range("asched_greedy_init");
  if (!params || !route_off || !route || !info) return ASCHED_E_INVALID;
  asched_params p0 = *params;
  p0.iterations = 0;
  p0.grid_clusters = 1;
  asched_result out = {};
  out.route_off = route_off;
  out.route = route;
  out.info = info;
  return asched_solve(inst, &p0, nullptr, nullptr, &out, stream);
}

int asched_tabu_solve(const asched_instance* inst, const asched_params* params, const int32_t* init_route_off,
                      const int32_t* init_route, const asched_result* out, void* workspace, size_t workspace_bytes,
                      void* stream) {
  const asched_nvtx::Range nvtx_range("asched_tabu_solve");
  if (!out || !out->route_off || !out->route || !out->info) return ASCHED_E_INVALID;
  if ((init_route_off == nullptr) != (init_route == nullptr)) return ASCHED_E_INVALID;
  return launch(inst, params, false, solve_params(init_route_off, init_route, out), workspace, workspace_bytes, true,
                stream);
}

int asched_batch_workspace_bytes(int32_t n_instances, size_t* out) {
  if (!out || n_instances < 0) return ASCHED_E_INVALID;
  *out = sizeof(int32_t) * (static_cast<size_t>(n_instances) + 1);
  return ASCHED_OK;
}

int asched_solve_batch(const asched_batch* batch, const asched_params* params, const asched_batch_result* out,
                       void* workspace, size_t workspace_bytes, void* stream) {
  const asched_nvtx::Range nvtx_range("asched_solve_batch");
  return launch_batch(batch, params, out, workspace, workspace_bytes, stream);
}

int asched_solve_batch_static(const asched_batch* batch, const asched_params* params,
                              const asched_batch_result* out, void* stream) {
  const asched_nvtx::Range nvtx_range("asched_solve_batch_static");
  if (!batch) return ASCHED_E_INVALID;
  if (batch->n_instances > ASCHED_STATIC_BATCH_MAX) return ASCHED_E_TOO_LARGE;
  void* scratch = nullptr;
  const int rc = static_scratch(&scratch);
  if (rc != ASCHED_OK) return rc;
  return launch_batch(batch, params, out, scratch, sizeof(g_batch_scratch), stream);
}

int asched_server_sizes(int32_t max_loc, int32_t max_vehicles, int32_t max_missions, int32_t n_types,
                        int32_t* slot_words, int32_t* out_words) {
  if (!slot_words || !out_words || max_loc < 1 || max_vehicles < 1 || max_missions < 0 || n_types < 1 ||
      n_types > 2)
    return ASCHED_E_INVALID;
  *slot_words = serve_slot_words(max_loc, max_vehicles, max_missions, n_types);
  *out_words = serve_out_words(max_vehicles, max_missions);
  return ASCHED_OK;
}

int asched_serve(const asched_server* server, const asched_params* params, int64_t idle_timeout_ns,
                 int32_t max_ctas, void* stream) {
  const asched_nvtx::Range nvtx_range("asched_serve");
  return launch_serve(server, params, idle_timeout_ns, max_ctas, stream);
}

int asched_eval_neighbourhood(const asched_instance* inst, const asched_params* params,
                              const int32_t* route_off, const int32_t* route, const int32_t* tabu_until,
                              int32_t it, int32_t z_best, int32_t* delta_out, uint8_t* flags_out,
                              uint32_t* id_out, unsigned long long* best_key_out, int32_t* info,
                              void* stream) {
  const asched_nvtx::Range nvtx_range("asched_eval_neighbourhood");
  if (!route_off || !route || !delta_out || !flags_out || !best_key_out || !info) return ASCHED_E_INVALID;
  KParams kp = {};
  kp.init_off = route_off;
  kp.init_route = route;
  kp.tabu_in = tabu_until;
  kp.dbg_it = it;
  kp.dbg_zbest = z_best;
  kp.dbg_delta = delta_out;
  kp.dbg_flags = flags_out;
  kp.dbg_id = id_out;
  kp.dbg_key = best_key_out;
  kp.info = info;
  return launch(inst, params, true, kp, nullptr, 0, false, stream);
}

}  // extern "C"
