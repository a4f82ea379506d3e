// Host runtime behind the C ABI of include/tpmc.h: contexts, resident meshes,
// memory admission, query set-up, launches and result read-back.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "runtime.h"

namespace tpmc {

thread_local std::string g_last_error;

tpmc_status fail(tpmc_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

tpmc_status cuda_fail(cudaError_t e, const char* where) {
  return fail(TPMC_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

// ------------------------------------------------------------ allocation
// take_pools: the pools of seeded particles give way when their memory is what is
// missing, which waits for the launches that use them.
tpmc_status Ctx::alloc(void** p, size_t bytes, const char* what, bool take_pools) {
  *p = nullptr;
  if (bytes == 0) return TPMC_OK;
  if (take_pools && used + bytes > budget && used + bytes <= budget + pooled()) release_pools();
  if (used + bytes > budget)
    return fail(TPMC_ENOMEM, std::string(what) + ": memory budget exceeded (" + std::to_string(used + bytes) +
                                 " > " + std::to_string(budget) + " bytes)");
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess && take_pools && release_pools()) {
    cudaGetLastError();
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return fail(TPMC_ENOMEM, std::string(what) + ": cudaMalloc: " + cudaGetErrorString(e));
  }
  sizes[*p] = bytes;
  used += bytes;
  ++n_allocs;
  return TPMC_OK;
}

void Ctx::release(void* p) {
  if (!p) return;
  auto it = sizes.find(p);
  if (it != sizes.end()) {
    used -= it->second;
    sizes.erase(it);
  }
  cudaFree(p);
}

tpmc_status Ctx::grow(Scratch& s, size_t bytes, const char* what) {
  if (s.cap >= bytes) return TPMC_OK;
  release(s.ptr);
  s.ptr = nullptr;
  s.cap = 0;
  size_t want = std::max(bytes, (size_t)256);
  tpmc_status st = alloc(&s.ptr, want, what);
  if (st == TPMC_OK) s.cap = want;
  return st;
}

// ---------------------------------------------------------------- params
tpmc_status validate_params(const tpmc_params* p) {
  if (!p) return fail(TPMC_EINVAL, "params is NULL");
  const double pos[] = {p->n, p->T_inf, p->m, p->V, p->T_W, p->A_ref};
  const char* names[] = {"n", "T_inf", "m", "V", "T_W", "A_ref"};
  for (int i = 0; i < 6; ++i)
    if (!(std::isfinite(pos[i]) && pos[i] > 0.0)) return fail(TPMC_EINVAL, std::string(names[i]) + " must be finite and > 0");
  if (!(p->eps_diffuse >= 0.0 && p->eps_diffuse <= 1.0)) return fail(TPMC_EINVAL, "eps_diffuse must be in [0, 1]");
  const double dn = std::sqrt(p->dir[0] * p->dir[0] + p->dir[1] * p->dir[1] + p->dir[2] * p->dir[2]);
  if (!(std::isfinite(dn) && dn > 0.0)) return fail(TPMC_EINVAL, "dir must be finite and non-zero");
  for (int i = 0; i < 3; ++i)
    if (!std::isfinite(p->ref_point[i]) || !std::isfinite(p->center[i])) return fail(TPMC_EINVAL, "non-finite point");
  if (!std::isfinite(p->r_cv)) return fail(TPMC_EINVAL, "r_cv must be finite");
  // the trace kernel keeps a particle's hit count in 24 bits beside its id
  if (p->max_bounces < 1 || p->max_bounces > (1u << 24) - 1)
    return fail(TPMC_EINVAL, "max_bounces must be in [1, 2^24 - 1]");
  if (p->precision != TPMC_FP32 && p->precision != TPMC_FP64) return fail(TPMC_EINVAL, "unknown precision");
  if (p->cv_kind > TPMC_CV_BOX_MAXWELL) return fail(TPMC_EINVAL, "unknown cv_kind");
  if (!std::isfinite(p->l_ref)) return fail(TPMC_EINVAL, "l_ref must be finite");
  if (p->gsi_model > TPMC_GSI_CLL) return fail(TPMC_EINVAL, "unknown gsi_model");
  if (p->gsi_model == TPMC_GSI_CLL &&
      !(p->alpha_n >= 0.0 && p->alpha_n <= 1.0 && p->sigma_t >= 0.0 && p->sigma_t <= 1.0))
    return fail(TPMC_EINVAL, "CLL: alpha_n and sigma_t must be in [0, 1]");
  if (p->cv_kind != TPMC_CV_SPHERE)
    for (int i = 0; i < 3; ++i)
      if (!(std::isfinite(p->box_lo[i]) && std::isfinite(p->box_hi[i]) && p->box_hi[i] > p->box_lo[i]))
        return fail(TPMC_EINVAL, "box CV: box_lo and box_hi must be finite with box_hi > box_lo");
  return TPMC_OK;
}

tpmc_status fill_query(const MeshRec& m, const tpmc_params* p, uint64_t N, QueryDev* q) {
  std::memset(q, 0, sizeof(*q));
  q->n = p->n; q->T_inf = p->T_inf; q->m = p->m; q->V = p->V;
  for (int i = 0; i < 3; ++i) { q->dir[i] = p->dir[i]; q->ref[i] = p->ref_point[i]; }
  q->T_W = p->T_W; q->eps = p->eps_diffuse; q->A_ref = p->A_ref;
  // The Maxwell choice u < eps on the uniform u = (k + 1/2) 2^-23 of a draw's
  // top 23 bits k holds exactly when k < eps 2^23 - 1/2, i.e. k < ceil(eps 2^23 - 1/2)
  // (eps 2^23 - 1/2 is exact in double), so the kernel decides in integers.
  q->eps_k = (uint32_t)std::min(8388608.0, std::max(0.0, std::ceil(p->eps_diffuse * 8388608.0 - 0.5)));
  q->l_ref = p->l_ref > 0.0 ? p->l_ref : 1.0;
  q->cv_kind = p->cv_kind;
  q->gsi_model = p->gsi_model;
  if (p->gsi_model == TPMC_GSI_CLL) {
    const double at = p->sigma_t * (2.0 - p->sigma_t);
    const double c[4] = {p->alpha_n, std::sqrt(1.0 - p->alpha_n), at, std::sqrt(std::max(0.0, 1.0 - at))};
    for (int i = 0; i < 4; ++i) { q->cll[i] = c[i]; q->fcll[i] = (float)c[i]; }
  }
  if (p->cv_kind != TPMC_CV_SPHERE) {
    // box CV: the body must lie strictly inside the box
    for (int i = 0; i < 3; ++i) {
      q->box_lo[i] = p->box_lo[i];
      q->box_hi[i] = p->box_hi[i];
      q->center[i] = 0.5 * (p->box_lo[i] + p->box_hi[i]);
    }
    q->r_cv = 0.0;
    for (int i = 0; i < 3 && !m.h_tri.empty(); ++i)
      if (!(m.lo[i] > q->box_lo[i] && m.hi[i] < q->box_hi[i]))
        return fail(TPMC_EINVAL, "the mesh is not strictly inside the box control volume");
  } else if (p->r_cv <= 0.0) {
    for (int i = 0; i < 3; ++i) q->center[i] = m.center[i];
    q->r_cv = m.radius > 0.0 ? 1.05 * m.radius : 1.0;
  } else {
    for (int i = 0; i < 3; ++i) q->center[i] = p->center[i];
    q->r_cv = p->r_cv;
    // the body must lie strictly inside the control volume: it does when its
    // bounding sphere does (to 1e-9); else its vertices decide (a pass of 0.2 ms
    // over 60,000 triangles and 2 ms over 500,000, once on every call)
    double apart2 = 0.0;
    for (int i = 0; i < 3; ++i) apart2 += (m.center[i] - q->center[i]) * (m.center[i] - q->center[i]);
    const bool inside = (std::sqrt(apart2) + m.radius) * (1.0 + 1e-9) < q->r_cv;
    double far2 = 0.0;
    for (uint64_t k = 0; !inside && k < m.h_tri.size(); ++k) {
      const double* v = &m.h_xyz[3 * (size_t)m.h_tri[k]];
      double d2 = 0.0;
      for (int i = 0; i < 3; ++i) d2 += (v[i] - q->center[i]) * (v[i] - q->center[i]);
      far2 = std::max(far2, d2);
    }
    if (!(std::sqrt(far2) < q->r_cv)) return fail(TPMC_EINVAL, "the mesh is not strictly inside the control volume");
  }
  double dref = 0.0;
  for (int i = 0; i < 3; ++i) dref += (m.center[i] - q->ref[i]) * (m.center[i] - q->ref[i]);
  q->rmax = std::sqrt(dref) + m.radius;
  q->N = N;
  q->seed = p->seed;
  q->stream_id = p->stream_id;
  q->max_bounces = p->max_bounces;
  q->precision = p->precision;
  q->panel = nullptr;
  return TPMC_OK;
}

LaunchCfg Ctx::schedule(const MeshRec& m, uint32_t variant, uint64_t total) {
  LaunchCfg cfg;
  const uint64_t key = tune_key(m.dev.n_tri, variant & ~kVariantPool);
  auto it = tuned.find(key);
  if (manual_launch) cfg = manual;
  else if (it != tuned.end()) cfg = it->second;
  else {
    // Untuned default, from same-box sweeps on GB300 with the current kernel
    // at 96 cases x 2e6 and x 1e7 particles per launch: 128 threads at the
    // highest occupancy (8 blocks per SM) for every tree.  Against 256 x 2
    // (no register cap) the plate is 4-8 % faster, the cylinder 25 %, the
    // satellite 23 %; against 6 blocks per SM the cylinder 9 % and the
    // satellite 10 % faster, the diffuse plate 0.6 % slower.
    cfg.block = 128;
    cfg.smem_nodes = 0;  // the hot top of the tree stays in L1; shared-memory staging costs bank conflicts
    cfg.blocks_per_sm = 0;
    cfg.chunk = 0;
    // Launches that 4 blocks per SM hold at once (77,824 particles on 152 SMs)
    // run the kernel without a register cap: 4,096 and 40,000 particles on the
    // hemisphere 276 -> 259 and 422 -> 386 us, on the satellite 136 -> 125 and
    // 199 -> 186; at 160,000 the two are equal, beyond more warps win.
    if (total > 0 && total <= (uint64_t)num_sms * 4 * 128 && (variant & 1u) == TPMC_FP32) cfg.blocks_per_sm = 4;
  }
  cfg.smem_nodes = m.dev.width > 2 ? 0u : std::min<uint32_t>(cfg.smem_nodes, m.dev.n_nodes);  // wide: none staged
  // the kernel's own fixed shared memory comes out of the largest staging
  size_t smem = trace_smem_bytes(cfg, m.dev.n_nodes, variant);
  if (smem <= 227 * 1024 && smem + kTraceStaticSmem > 227 * 1024) cfg.smem_nodes -= kTraceStaticSmem / 32;
  smem = trace_smem_bytes(cfg, m.dev.n_nodes, variant);
  // A traversal round ends once this many lanes have finished their rays.
  // Same-box sweeps with the current kernel: 16 to 28 are equal on the plate
  // and the cylinder; on the satellite 16 is 3 % faster than 24 and 2 % than 20.
  if (cfg.refill_at == 0 || cfg.refill_at > 32) cfg.refill_at = 16;
  // asked of the driver once for each kernel and block (10 us a time)
  auto occ = max_blocks.emplace(((uint64_t)smem << 32) | ((uint64_t)variant << 16) | cfg.block, 0);
  if (occ.second) occ.first->second = trace_max_blocks_per_sm(variant, cfg, m.dev.n_nodes);
  const int maxb = occ.first->second;
  if (cfg.blocks_per_sm == 0 || (int)cfg.blocks_per_sm > maxb) cfg.blocks_per_sm = std::max(1, maxb);
  if (cfg.chunk == 0) {
    const uint64_t warps = (uint64_t)num_sms * cfg.blocks_per_sm * (cfg.block / 32);
    uint64_t ch = total / std::max<uint64_t>(1, warps * 16);
    ch = (ch / 32) * 32;
    cfg.chunk = (uint32_t)std::min<uint64_t>(1024, std::max<uint64_t>(32, ch));
    // fewer particles than lanes: an equal share for every warp, so that the
    // lanes of a warp wait for fewer others (1,000 and 16,000 particles on the
    // hemisphere 336 -> 214 and 447 -> 335 us, 4,096 on the icosphere 105 -> 91)
    const uint64_t share = (total + warps - 1) / std::max<uint64_t>(1, warps);
    if (share > 0 && share < 32) cfg.chunk = (uint32_t)share;
  }
  return cfg;
}

// Mean projected area over pi, m^2, of a query's control volume.
float cv_area(const QueryDev& q) {
  if (q.cv_kind == TPMC_CV_SPHERE) return (float)(q.r_cv * q.r_cv);
  const double x = q.box_hi[0] - q.box_lo[0], y = q.box_hi[1] - q.box_lo[1], z = q.box_hi[2] - q.box_lo[2];
  return (float)((x * y + y * z + z * x) / 6.283185307179586);
}

// A pool for launches of `total` particles in batches of at most max_batch, in the
// memory the context's budget leaves (pool_entries); false when it has no room (the
// launch then seeds inside the trace kernel).  A pool outlives its call, so a new one
// also takes at most a quarter of the device's free memory: three quarters stay for
// whoever shares the device and cannot ask for the pool back.
bool Ctx::grow_pool(Pool& pool, uint64_t total, uint64_t max_batch) {
  pool.max_batch = max_batch;
  size_t room = budget - std::min(budget, used - pool.cap);
  uint64_t entries = pool_entries(total, max_batch, room);
  if (entries > 0 && pool.cap < pool_bytes(entries)) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    room = std::min(room, (free_b + pool.cap) / 2);
    entries = pool_entries(total, max_batch, room);
  }
  if (entries == 0) return false;
  const size_t need = pool_bytes(entries);
  if (pool.cap >= need) return true;
  release_pool(pool);
  const std::string last = g_last_error;
  if (alloc(&pool.ptr, need, "seeded particles", false) == TPMC_OK) {
    pool.cap = need;
    return true;
  }
  g_last_error = last;  // not the caller's failure
  return false;
}

// Frees a pool once the kernels that use it are done.
void Ctx::release_pool(Pool& pool) {
  if (!pool.ptr) return;
  if (pool.done) cudaEventSynchronize(pool.done);
  release(pool.ptr);
  pool.ptr = nullptr;
  pool.cap = 0;
}

// Pools give way to everything else that needs the memory (Ctx::alloc, where it helps).
bool Ctx::release_pools() {
  bool any = false;
  for (Pool* p : pools) {
    any = any || p->ptr;
    release_pool(*p);
  }
  return any;
}

size_t Ctx::pooled() const {
  size_t n = 0;
  for (const Pool* p : pools) n += p->cap;
  return n;
}

void Ctx::destroy_pool(Pool& pool) {
  release_pool(pool);
  if (pool.side) cudaStreamDestroy(pool.side);
  for (cudaEvent_t ev : {pool.fork, pool.join, pool.done})
    if (ev) cudaEventDestroy(ev);
  pool = Pool();
}

// Traces a launch through the pool: in one batch, or in batches of half of it,
// seed_kernel then trace_kernel, in turn on the context's stream and on a second
// one, which joins it again at the end.  A batch ends in a tail of its longest
// paths (up to 0.6 ms on the satellite: 64 bounces, one after the other); the other
// stream's next kernels fill it.  One stream and batches of 2^26, 2^27 particles:
// the attitude sweep 236 and 226 ms; two streams of 2^26: 217 (of 2^27: 211, for
// twice the memory).
// a.counter: kRunCounters counters.  Particles beyond max_batches batches are traced
// by one launch that seeds them itself.
cudaError_t Ctx::trace_pool(Pool& pool, cudaStream_t stream, TraceArgs a, uint32_t variant, const LaunchCfg& cfg,
                            const MeshRec& m, float area, uint64_t max_batches) {
  // Rough rays first where less than 45 % of the particles are expected to meet
  // the front (its mean projected area over the control volume's).  They cost
  // 55 % of an exact seeding and what passes is seeded exactly after them: the
  // satellite (12 % pass) 6.74 -> 6.09 ms for 1e8 particles, the plate sweep
  // (36 %) 32.7 -> 31.6; the cylinder's (55 %) would take 94.9 for 92.9, so it
  // seeds exactly at once.
  a.prefilter = a.mesh.front_area < 0.45f * area ? 1u : 0u;
  cudaError_t e = cudaSuccess;
  if (!pool.side) e = cudaStreamCreateWithFlags(&pool.side, cudaStreamNonBlocking);
  for (cudaEvent_t* ev : {&pool.fork, &pool.join, &pool.done})
    if (e == cudaSuccess && !*ev) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
  if (e != cudaSuccess) return e;
  uint64_t total = a.total;
  const uint64_t entries = (pool.cap - pool_bytes(0)) / (32 * kPoolEntryBytes + sizeof(uint32_t)) * 32;
  uint64_t batch = pool_batch(entries, total, pool.max_batch);
  // Segments of 32 to 2,048 work indices (a power of two): as long as the trace
  // grid still gets eight a warp to even out its work, or two behind rough rays,
  // where few particles of a segment pass.  Every segment costs a fetch, and behind
  // rough rays an exact seeding with lanes idle for its last candidates.  At most
  // 512 and eight a warp always -> now: plate sweep 31.5 -> 30.3 ms, cylinder sweep
  // 91.8 -> 90.8, attitude sweep 185.5 -> 177.9, 1e7 particles on the
  // 500,000-triangle satellite 1,353 -> 1,277 us (at most 4,096: 30.4, -, 178.8,
  // 1,275; four a warp on the hemisphere, without rough rays, 6.67 ms for 6.55).
  const uint64_t warps = (uint64_t)num_sms * cfg.blocks_per_sm * (cfg.block / 32);
  const uint64_t per_warp = std::min(batch, total) / ((a.prefilter ? 2 : 8) * std::max<uint64_t>(1, warps));
  a.segment = 32;
  while (2 * a.segment <= per_warp && a.segment < kPoolSegment) a.segment *= 2;
  batch = batch / a.segment * a.segment;
  if (max_batches < total / batch) total = max_batches * batch;
  bool forked = false;
  uint64_t i = 0;
  for (a.g0 = 0; a.g0 < total && e == cudaSuccess; a.g0 += batch, ++i) {
    const bool side = (i & 1) != 0;
    if (side && !forked) {
      // the second stream starts where the set-up left the first
      if ((e = cudaStreamWaitEvent(pool.side, pool.fork, 0)) != cudaSuccess) break;
      forked = true;
    }
    if (i == 0 && total > batch && (e = cudaEventRecord(pool.fork, stream)) != cudaSuccess) break;
    TraceArgs b = a;
    b.total = std::min(total, a.g0 + batch);
    b.n_seg = (uint32_t)((b.total - a.g0 + a.segment - 1) / a.segment);
    char* half = (char*)pool.ptr + (side ? (pool.cap / 2) & ~(size_t)255 : 0);
    b.pool = half;
    b.seg_count = (uint32_t*)(half + batch * kPoolEntryBytes);
    b.counter = a.counter + (side ? 1 : 0);
    const cudaStream_t st = side ? pool.side : stream;
    if ((e = launch_seed(b, st)) == cudaSuccess) e = launch_trace(b, variant, cfg, num_sms, st);
  }
  if (forked) {  // also after an error: what was enqueued ends before anything else on the stream
    cudaError_t e2 = cudaEventRecord(pool.join, pool.side);
    if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(stream, pool.join, 0);
    if (e == cudaSuccess) e = e2;
  }
  const cudaError_t e3 = cudaEventRecord(pool.done, stream);
  if (e == cudaSuccess) e = e3;
  if (e == cudaSuccess && total < a.total) {
    TraceArgs r = a;
    r.pool = nullptr;
    r.g0 = total;
    r.counter = a.counter + kRunCounters - 1;
    const LaunchCfg c = schedule(m, variant & ~kVariantPool, a.total - total);
    r.chunk = c.chunk;
    r.smem_nodes = c.smem_nodes;
    r.refill_at = c.refill_at;
    e = launch_trace(r, variant & ~kVariantPool, c, num_sms, stream);
  }
  return e;
}

// One batched run: nq queries prepared on the device from `base` (+ dirs/S),
// traced together, finalised into d_out (device memory or the context's pinned
// results).  Three launches and no copies: the base query goes with the set-up's
// launch, which also clears the counters, and the reduction writes the error
// word to pinned memory (two uploads, a memset and two downloads took 25 us of
// a small call).
tpmc_status Ctx::run(const MeshRec& m, uint32_t nq, const QueryDev& base, const double* d_dirs, const double* d_S,
                     uint64_t total, uint32_t variant, tpmc_result* d_out, const RecordsDev* rec, uint64_t max_batches) {
  tpmc_status st;
  if ((st = grow(s_queries, sizeof(QueryDev) * (size_t)nq, "queries")) != TPMC_OK) return st;
  if ((st = grow(s_acc, sizeof(AccStripe) * kAccStripes * (size_t)nq, "accumulators")) != TPMC_OK) return st;
  if ((st = grow(s_items, sizeof(ItemDev) * (size_t)nq, "work items")) != TPMC_OK) return st;
  if ((st = grow(s_misc, sizeof(RunWords), "counters")) != TPMC_OK) return st;
  QueryDev* d_queries = (QueryDev*)s_queries.ptr;
  AccStripe* d_acc = (AccStripe*)s_acc.ptr;
  ItemDev* d_items = (ItemDev*)s_items.ptr;
  RunWords* words = (RunWords*)s_misc.ptr;
  cudaError_t e;
  // the set-up also clears the queries' accumulators
  if ((e = launch_setup(d_queries, nq, &base, d_dirs, d_S, d_items, nullptr, d_acc, nq, vn_table, words, num_sms,
                        stream)) != cudaSuccess)
    return cuda_fail(e, "setup kernel");
  TraceArgs a{};
  a.mesh = m.dev;
  a.queries = d_queries;
  a.acc = d_acc;
  a.acc_stride = nq;
  a.items = d_items;
  a.n_items = nq;
  a.total = total;
  a.counter = words->counter;
  a.error = &words->error;
  a.count_work = counters ? 1u : 0u;
  a.vn_table = vn_table;
  if (rec) a.rec = *rec;
  const bool pooled = !counters && !rec && (variant & 1u) == TPMC_FP32 && total > 0 &&
                      (pool_always || total >= kPoolMin) && grow_pool(pool, total, kPoolBatch);
  if (pooled) variant |= kVariantPool;
  const LaunchCfg cfg = schedule(m, variant, total);
  a.chunk = cfg.chunk;
  a.smem_nodes = cfg.smem_nodes;
  a.refill_at = cfg.refill_at;
  last_cfg = cfg;
  if (total > 0 && (e = pooled ? trace_pool(pool, stream, a, variant, cfg, m, cv_area(base), max_batches)
                               : launch_trace(a, variant, cfg, num_sms, stream)) != cudaSuccess)
    return cuda_fail(e, "trace kernel");
  if ((e = launch_finalize(d_queries, d_acc, nq, nq, nullptr, d_out, &words->error, h_err_word, stream)) != cudaSuccess)
    return cuda_fail(e, "finalize kernel");
  return TPMC_OK;
}

tpmc_status Ctx::check_error_word() {
  if (*h_err_word != 0) {
    const int w = *h_err_word;
    *h_err_word = 0;
    return fail(TPMC_ECUDA, "trace kernel reported error word " + std::to_string(w) + " (traversal stack overflow)");
  }
  return TPMC_OK;
}

// BVH width of a mesh load: the one set by tpmc_set_launch, else the one
// tpmc_tune chose for the size class, else the default.
uint32_t Ctx::width_for(uint32_t n_tri) const {
  if (bvh_width) return bvh_width;
  auto it = tuned_width.find(tune_key(n_tri, 0));
  return it != tuned_width.end() ? it->second : kDefaultBvhWidth;
}

// Builds the mesh's BVH with `width` children per node and uploads it, its
// triangles and frames into one device allocation (the host copies of the
// mesh are not set here).
tpmc_status Ctx::upload_mesh(const double* xyz, uint32_t n_vert, const uint32_t* tri, uint32_t n_tri, uint32_t width,
                             MeshRec* out) {
  BvhBuild b;
  const char* err = nullptr;
  if (!build_bvh(xyz, n_vert, tri, n_tri, bvh_leaf, width, &b, &err)) {
    b.release();
    return fail(TPMC_EINVAL, err);
  }
  MeshRec& m = *out;
  const size_t sz_nodes = b.n_nodes * b.node_bytes;
  const size_t sz_tris = (size_t)b.n_leaf_tris * 12 * sizeof(float);
  const size_t sz_tris64 = (size_t)b.n_leaf_tris * 12 * sizeof(double);
  const size_t sz_fr = (size_t)n_tri * 8 * sizeof(float);
  const size_t sz_fr64 = (size_t)n_tri * 8 * sizeof(double);
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t total = al(sz_nodes) + al(sz_tris) + al(sz_tris64) + al(sz_fr) + al(sz_fr64);
  tpmc_status st = alloc(&m.d_block, std::max(total, (size_t)256), "mesh");
  if (st != TPMC_OK) { b.release(); return st; }
  char* base = (char*)m.d_block;
  size_t off = 0;
  auto place = [&](size_t sz) { char* p = base + off; off += al(sz); return p; };
  char* p_nodes = place(sz_nodes);
  char* p_tris = place(sz_tris);
  char* p_tris64 = place(sz_tris64);
  char* p_fr = place(sz_fr);
  char* p_fr64 = place(sz_fr64);
  cudaError_t e = cudaSuccess;
  if (sz_nodes) e = cudaMemcpy(p_nodes, b.nodes, sz_nodes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && sz_tris) e = cudaMemcpy(p_tris, b.tris, sz_tris, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && sz_tris64) e = cudaMemcpy(p_tris64, b.tris64, sz_tris64, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && sz_fr) e = cudaMemcpy(p_fr, b.frames, sz_fr, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && sz_fr64) e = cudaMemcpy(p_fr64, b.frames64, sz_fr64, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    release(m.d_block);
    m.d_block = nullptr;
    b.release();
    return cuda_fail(e, "upload mesh");
  }
  m.dev.nodes = (const float4*)p_nodes;
  m.dev.tris = (const float4*)p_tris;
  m.dev.tris64 = (const double*)p_tris64;
  m.dev.frames = (const float4*)p_fr;
  m.dev.frames64 = (const double*)p_fr64;
  m.dev.n_nodes = (uint32_t)b.n_nodes;
  m.dev.width = b.width;
  m.dev.depth = b.depth;
  for (int k = 0; k < 3; ++k) {
    m.dev.qorigin[k] = b.qorigin[k];
    m.dev.qstep[k] = b.qstep[k];
    m.dev.qinv[k] = 1.0f / b.qstep[k];
  }
  m.dev.n_front = b.n_front;
  m.dev.front_area = b.front_area;
  std::memcpy(m.dev.front_reach, b.front_reach, sizeof(b.front_reach));
  std::memcpy(m.dev.front, b.front, sizeof(b.front));
  m.dev.n_tri = n_tri;
  m.dev.n_tri_leaf = b.n_leaf_tris;
  m.dev.scene_radius = (float)b.radius;
  for (int i = 0; i < 3; ++i) m.dev.centre[i] = (float)b.center[i];
  for (int i = 0; i < 3; ++i) m.center[i] = b.center[i];
  m.radius = b.radius;
  for (int i = 0; i < 3; ++i) { m.lo[i] = b.lo[i]; m.hi[i] = b.hi[i]; }
  m.depth = b.depth;
  m.leaf_max = b.leaf_max;
  m.n_skipped = b.n_skipped;
  m.n_exposed = b.n_exposed;
  m.node_bytes = b.node_bytes;
  m.n_vert = n_vert;
  m.bytes = total;
  b.release();
  return TPMC_OK;
}

Ctx::~Ctx() {
  if (serve) stop_serving(this);
  for (auto& kv : panels) release(kv.second.d_panel);
  for (auto& kv : meshes) release(kv.second.d_block);
  for (Scratch* s : {&s_queries, &s_acc, &s_items, &s_misc, &s_out, &s_in})
    release(s->ptr);
  release(vn_table);
  if (h_pinned) cudaFreeHost(h_pinned);
  destroy_pool(pool);
  if (own_stream) cudaStreamDestroy(own_stream);
}

}  // namespace tpmc

using namespace tpmc;

// =========================================================================
extern "C" {

tpmc_status tpmc_create(int device, size_t mem_budget_bytes, tpmc_ctx** out) {
  if (!out) return fail(TPMC_EINVAL, "out is NULL");
  *out = nullptr;
  int n = 0;
  cudaError_t e = cudaGetDeviceCount(&n);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceCount");
  if (device < 0 || device >= n) return fail(TPMC_EINVAL, "no such CUDA device");
  if ((e = cudaSetDevice(device)) != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
  std::unique_ptr<Ctx> c(new Ctx());
  c->device = device;
  cudaDeviceProp prop;
  if ((e = cudaGetDeviceProperties(&prop, device)) != cudaSuccess) return cuda_fail(e, "cudaGetDeviceProperties");
  c->num_sms = prop.multiProcessorCount;
  size_t free_b = 0, total_b = 0;
  if ((e = cudaMemGetInfo(&free_b, &total_b)) != cudaSuccess) return cuda_fail(e, "cudaMemGetInfo");
  c->budget = mem_budget_bytes ? mem_budget_bytes : (size_t)(0.9 * (double)free_b);
  if ((e = cudaStreamCreateWithFlags(&c->own_stream, cudaStreamNonBlocking)) != cudaSuccess)
    return cuda_fail(e, "cudaStreamCreate");
  c->stream = c->own_stream;
  if ((e = cudaMallocHost(&c->h_pinned, kPinnedBytes)) != cudaSuccess) return cuda_fail(e, "cudaMallocHost");
  {
    void* t = nullptr;
    tpmc_status st = c->alloc(&t, sizeof(float) * kTableFloats, "start tables");
    if (st != TPMC_OK) return st;
    c->vn_table = (float*)t;
    if ((e = launch_tables(c->vn_table, c->stream)) != cudaSuccess) return cuda_fail(e, "start tables");
    if ((e = cudaStreamSynchronize(c->stream)) != cudaSuccess) return cuda_fail(e, "start tables");
  }
  c->h_err_word = (int*)c->h_pinned;
  c->h_results = (tpmc_result*)((char*)c->h_pinned + 256);
  c->h_inputs = (double*)((char*)c->h_pinned + 256 + kPinnedItems * sizeof(tpmc_result));
  *c->h_err_word = 0;
  *out = reinterpret_cast<tpmc_ctx*>(c.release());
  return TPMC_OK;
}

tpmc_status tpmc_destroy(tpmc_ctx* ctx) {
  if (!ctx) return TPMC_OK;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  cudaSetDevice(c->device);
  cudaStreamSynchronize(c->stream);
  delete c;
  return TPMC_OK;
}

tpmc_status tpmc_set_stream(tpmc_ctx* ctx, void* cuda_stream) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  c->stream = cuda_stream ? (cudaStream_t)cuda_stream : c->own_stream;
  return TPMC_OK;
}

const char* tpmc_last_error(const tpmc_ctx*) { return g_last_error.c_str(); }

tpmc_status tpmc_memory_info(tpmc_ctx* ctx, size_t* used, size_t* budget, uint64_t* n_allocs) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  if (used) *used = c->used;
  if (budget) *budget = c->budget;
  if (n_allocs) *n_allocs = c->n_allocs;
  return TPMC_OK;
}

tpmc_status tpmc_set_counters(tpmc_ctx* ctx, int enable) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  c->counters = enable != 0;
  return TPMC_OK;
}

tpmc_status tpmc_mesh_load(tpmc_ctx* ctx, const double* xyz, uint32_t n_vert, const uint32_t* tri, uint32_t n_tri,
                           tpmc_mesh_id* out) {
  if (!ctx || !out) return fail(TPMC_EINVAL, "NULL argument");
  if ((n_vert > 0 && !xyz) || (n_tri > 0 && !tri)) return fail(TPMC_EINVAL, "NULL mesh array");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  cudaSetDevice(c->device);
  MeshRec m;
  tpmc_status st = c->upload_mesh(xyz, n_vert, tri, n_tri, c->width_for(n_tri), &m);
  if (st != TPMC_OK) return st;
  m.h_xyz.assign(xyz, xyz + 3 * (size_t)n_vert);
  m.h_tri.assign(tri, tri + 3 * (size_t)n_tri);
  const tpmc_mesh_id id = c->next_mesh++;
  c->meshes[id] = std::move(m);
  *out = id;
  return TPMC_OK;
}

tpmc_status tpmc_mesh_unload(tpmc_ctx* ctx, tpmc_mesh_id mesh) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  auto it = c->meshes.find(mesh);
  if (it == c->meshes.end()) return fail(TPMC_ENOTFOUND, "unknown mesh id");
  if (it->second.in_use > 0) return fail(TPMC_EBUSY, "mesh is used by queries in flight");
  cudaSetDevice(c->device);
  cudaStreamSynchronize(c->stream);
  c->release(it->second.d_block);
  c->meshes.erase(it);
  return TPMC_OK;
}

tpmc_status tpmc_mesh_info(tpmc_ctx* ctx, tpmc_mesh_id mesh, tpmc_mesh_stats* out) {
  if (!ctx || !out) return fail(TPMC_EINVAL, "NULL argument");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  auto it = c->meshes.find(mesh);
  if (it == c->meshes.end()) return fail(TPMC_ENOTFOUND, "unknown mesh id");
  const MeshRec& m = it->second;
  std::memset(out, 0, sizeof(*out));
  out->n_tri = m.dev.n_tri;
  out->n_vert = m.n_vert;
  out->n_nodes = m.dev.n_nodes;
  out->depth = m.depth;
  out->n_skipped = m.n_skipped;
  out->leaf_max = m.leaf_max;
  for (int i = 0; i < 3; ++i) out->bound_center[i] = m.center[i];
  out->bound_radius = m.radius;
  out->device_bytes = m.bytes;
  out->n_refs = m.dev.n_tri_leaf;
  out->n_exposed = m.n_exposed;
  out->bvh_width = m.dev.width;
  out->node_bytes = m.node_bytes;
  return TPMC_OK;
}

static tpmc_status trace_common(Ctx* c, tpmc_mesh_id mesh, const tpmc_params* params, uint64_t N,
                                tpmc_records* records, tpmc_result* out) {
  if (!out) return fail(TPMC_EINVAL, "out is NULL");
  tpmc_status st = validate_params(params);
  if (st != TPMC_OK) return st;
  if (N == 0 || N > (1ull << 34)) return fail(TPMC_EINVAL, "N must be in [1, 2^34]");
  auto it = c->meshes.find(mesh);
  if (it == c->meshes.end()) return fail(TPMC_ENOTFOUND, "unknown mesh id");
  const MeshRec& m = it->second;
  cudaSetDevice(c->device);
  const auto t0 = std::chrono::steady_clock::now();
  QueryDev q;
  if ((st = fill_query(m, params, N, &q)) != TPMC_OK) return st;
  // per-triangle loads
  void* d_panel = nullptr;
  if (params->want_panels && m.dev.n_tri > 0) {
    if ((st = c->alloc(&d_panel, (size_t)m.dev.n_tri * 3 * sizeof(long long), "panel loads")) != TPMC_OK) return st;
    cudaMemsetAsync(d_panel, 0, (size_t)m.dev.n_tri * 3 * sizeof(long long), c->stream);
    q.panel = (long long*)d_panel;
  }
  // records
  RecordsDev rec;
  void* d_rec = nullptr;
  if (records) {
    if (records->K > (uint32_t)kMaxRecordK || N > (1ull << 26)) {
      c->release(d_panel);
      return fail(TPMC_EINVAL, "records: K must be <= 64 and N <= 2^26");
    }
    const size_t K = std::max<uint32_t>(records->K, 1);
    const size_t bytes = N * (9 * sizeof(double) + (2 + K) * sizeof(uint32_t));
    if ((st = c->alloc(&d_rec, bytes, "records")) != TPMC_OK) { c->release(d_panel); return st; }
    char* p = (char*)d_rec;
    rec.pos = (double*)p; p += N * 3 * sizeof(double);
    rec.vel = (double*)p; p += N * 3 * sizeof(double);
    rec.dv = (double*)p; p += N * 3 * sizeof(double);
    rec.n_hits = (uint32_t*)p; p += N * sizeof(uint32_t);
    rec.truncated = (uint32_t*)p; p += N * sizeof(uint32_t);
    rec.tri = (uint32_t*)p;
    rec.K = records->K;
    cudaMemsetAsync(rec.tri, 0xFF, N * K * sizeof(uint32_t), c->stream);
  }
  const tpmc_status rs = c->run(m, 1, q, nullptr, nullptr, N, trace_variant(params, m.dev), c->h_results,
                                records ? &rec : nullptr);
  cudaError_t e = cudaSuccess;
  if (rs == TPMC_OK && e == cudaSuccess && records) {
    const size_t K = records->K;
    auto cp = [&](void* dst, const void* src, size_t bytes) {
      if (dst && e == cudaSuccess) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, c->stream);
    };
    cp(records->pos, rec.pos, N * 3 * sizeof(double));
    cp(records->vel, rec.vel, N * 3 * sizeof(double));
    cp(records->dv, rec.dv, N * 3 * sizeof(double));
    cp(records->n_hits, rec.n_hits, N * sizeof(uint32_t));
    cp(records->truncated, rec.truncated, N * sizeof(uint32_t));
    if (K) cp(records->tri, rec.tri, N * K * sizeof(uint32_t));
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (d_rec) c->release(d_rec);
  if (rs != TPMC_OK || e != cudaSuccess) {
    c->release(d_panel);
    return rs != TPMC_OK ? rs : cuda_fail(e, "trace");
  }
  if ((st = c->check_error_word()) != TPMC_OK) { c->release(d_panel); return st; }
  *out = *c->h_results;
  const auto t1 = std::chrono::steady_clock::now();
  out->ms = std::chrono::duration<double, std::milli>(t1 - t0).count();
  if (out->status != TPMC_OK) {
    c->release(d_panel);
    return fail((tpmc_status)out->status, "query set-up rejected the parameters (S outside [0.01, 50] or fixed-point range)");
  }
  out->query_id = c->next_query++;
  if (d_panel) {
    PanelRec pr;
    pr.d_panel = d_panel;
    pr.query = q;
    pr.mesh = mesh;
    pr.n_tri = m.dev.n_tri;
    // keep the set-up values the panel conversion needs
    pr.query.gamma = out->gamma;
    pr.query.m = params->m;
    pr.query.c_mp = out->c_mp;
    pr.query.quantum = out->fixed_quantum;
    c->panels[out->query_id] = pr;
  }
  return TPMC_OK;
}

tpmc_status tpmc_trace(tpmc_ctx* ctx, tpmc_mesh_id mesh, const tpmc_params* params, uint64_t N, tpmc_result* out) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  return trace_common(c, mesh, params, N, nullptr, out);
}

tpmc_status tpmc_trace_records(tpmc_ctx* ctx, tpmc_mesh_id mesh, const tpmc_params* params, uint64_t N,
                               tpmc_records* records, tpmc_result* out) {
  if (!ctx || !records) return fail(TPMC_EINVAL, "NULL argument");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  return trace_common(c, mesh, params, N, records, out);
}

static tpmc_status panels_locked(Ctx* c, tpmc_query_id query, double* pressure, double* shear, uint32_t n_tri) {
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  auto it = c->panels.find(query);
  if (it == c->panels.end()) return fail(TPMC_ENOTFOUND, "no panel loads kept for this query");
  PanelRec& pr = it->second;
  if (n_tri != pr.n_tri) return fail(TPMC_EINVAL, "n_tri does not match the mesh");
  auto mit = c->meshes.find(pr.mesh);
  if (mit == c->meshes.end()) return fail(TPMC_ENOTFOUND, "the query's mesh was unloaded");
  cudaSetDevice(c->device);
  tpmc_status st;
  if ((st = c->grow(c->s_in, sizeof(QueryDev), "panel query")) != TPMC_OK) return st;
  void* d_pv = nullptr;
  if ((st = c->alloc(&d_pv, (size_t)n_tri * 2 * sizeof(double), "panel output")) != TPMC_OK) return st;
  double* d_p = (double*)d_pv;
  double* d_s = d_p + n_tri;
  cudaError_t e = cudaMemcpyAsync(c->s_in.ptr, &pr.query, sizeof(QueryDev), cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess)
    e = launch_panels((const QueryDev*)c->s_in.ptr, (const long long*)pr.d_panel, mit->second.dev.frames,
                      mit->second.dev.frames64, n_tri, d_p, d_s, c->stream);
  if (e == cudaSuccess && pressure) e = cudaMemcpyAsync(pressure, d_p, n_tri * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess && shear) e = cudaMemcpyAsync(shear, d_s, n_tri * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  c->release(d_pv);
  if (e != cudaSuccess) return cuda_fail(e, "panels");
  c->release(pr.d_panel);
  c->panels.erase(it);
  return TPMC_OK;
}

tpmc_status tpmc_panels(tpmc_ctx* ctx, tpmc_query_id query, double* pressure, double* shear, uint32_t n_tri) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  const tpmc_status st = panels_locked(c, query, pressure, shear, n_tri);
  // after the context lock is dropped (the scheduler takes its own lock first)
  if (st == TPMC_OK) serve_memory_released(c);
  return st;
}

tpmc_status tpmc_panel_sums(tpmc_ctx* ctx, tpmc_query_id query, int64_t* dv_q, uint32_t n_tri) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!dv_q) return fail(TPMC_EINVAL, "dv_q is NULL");
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  auto it = c->panels.find(query);
  if (it == c->panels.end()) return fail(TPMC_ENOTFOUND, "no panel loads kept for this query");
  const PanelRec& pr = it->second;
  if (n_tri != pr.n_tri) return fail(TPMC_EINVAL, "n_tri does not match the mesh");
  cudaSetDevice(c->device);
  cudaError_t e = cudaMemcpyAsync(dv_q, pr.d_panel, (size_t)n_tri * 3 * sizeof(long long), cudaMemcpyDeviceToHost,
                                  c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(e, "panel sums");
  return TPMC_OK;
}

static tpmc_status sweep_common(Ctx* c, tpmc_mesh_id mesh, const tpmc_params* base, const double* d_dirs,
                                const double* d_S, uint32_t K, uint64_t N_each, tpmc_result* d_out,
                                uint64_t max_batches = ~0ull) {
  tpmc_status st = validate_params(base);
  if (st != TPMC_OK) return st;
  if (K == 0 || K > kMaxLaunchQueries) return fail(TPMC_EINVAL, "K must be in [1, 2^24]");
  if (N_each == 0 || N_each > (1ull << 34)) return fail(TPMC_EINVAL, "N_each must be in [1, 2^34]");
  if ((uint64_t)K * N_each > (1ull << 50)) return fail(TPMC_EINVAL, "K * N_each too large");
  auto it = c->meshes.find(mesh);
  if (it == c->meshes.end()) return fail(TPMC_ENOTFOUND, "unknown mesh id");
  const MeshRec& m = it->second;
  QueryDev q;
  if ((st = fill_query(m, base, N_each, &q)) != TPMC_OK) return st;
  return c->run(m, K, q, d_dirs, d_S, (uint64_t)K * N_each, trace_variant(base, m.dev), d_out, nullptr, max_batches);
}

tpmc_status tpmc_sweep(tpmc_ctx* ctx, tpmc_mesh_id mesh, const tpmc_params* base, const double* h_dirs,
                       const double* h_S, uint32_t K, uint64_t N_each, tpmc_result* h_out) {
  if (!ctx || !h_out) return fail(TPMC_EINVAL, "NULL argument");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  cudaSetDevice(c->device);
  const auto t0 = std::chrono::steady_clock::now();
  tpmc_status st;
  // Short sweeps: the kernels read their inputs from and write their results to
  // pinned memory; long ones go through device memory.
  const bool pinned = K <= kPinnedItems;
  double* d_in = c->h_inputs;
  tpmc_result* d_out = c->h_results;
  if (!pinned) {
    if ((st = c->grow(c->s_in, std::max((size_t)K * 4 * sizeof(double), sizeof(QueryDev)), "sweep inputs")) != TPMC_OK) return st;
    if ((st = c->grow(c->s_out, (size_t)K * sizeof(tpmc_result), "sweep results")) != TPMC_OK) return st;
    d_in = (double*)c->s_in.ptr;
    d_out = (tpmc_result*)c->s_out.ptr;
  }
  double* d_dirs = h_dirs ? d_in : nullptr;
  double* d_S = h_S ? d_in + 3 * (size_t)K : nullptr;
  cudaError_t e = cudaSuccess;
  if (pinned) {
    if (h_dirs) std::memcpy(d_dirs, h_dirs, (size_t)K * 3 * sizeof(double));
    if (h_S) std::memcpy(d_S, h_S, (size_t)K * sizeof(double));
  } else {
    if (h_dirs) e = cudaMemcpyAsync(d_dirs, h_dirs, (size_t)K * 3 * sizeof(double), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess && h_S) e = cudaMemcpyAsync(d_S, h_S, (size_t)K * sizeof(double), cudaMemcpyHostToDevice, c->stream);
    if (e != cudaSuccess) return cuda_fail(e, "upload sweep inputs");
  }
  if ((st = sweep_common(c, mesh, base, d_dirs, d_S, K, N_each, d_out)) != TPMC_OK) return st;
  if (!pinned) e = cudaMemcpyAsync(h_out, d_out, (size_t)K * sizeof(tpmc_result), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(e, "sweep");
  if ((st = c->check_error_word()) != TPMC_OK) return st;
  if (pinned) std::memcpy(h_out, d_out, (size_t)K * sizeof(tpmc_result));
  const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  for (uint32_t k = 0; k < K; ++k) h_out[k].ms = ms;
  return TPMC_OK;
}

tpmc_status tpmc_sweep_device(tpmc_ctx* ctx, tpmc_mesh_id mesh, const tpmc_params* base, const double* d_dirs,
                              const double* d_S, uint32_t K, uint64_t N_each, tpmc_result* d_out) {
  if (!ctx || !d_out) return fail(TPMC_EINVAL, "NULL argument");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  cudaSetDevice(c->device);
  return sweep_common(c, mesh, base, d_dirs, d_S, K, N_each, d_out, kPoolBatchesQueued);
}

tpmc_status tpmc_set_launch(tpmc_ctx* ctx, const tpmc_launch* cfg) {
  if (!ctx) return fail(TPMC_EINVAL, "ctx is NULL");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  if (!cfg) {
    c->manual_launch = false;
    c->bvh_leaf = 4;
    c->bvh_width = 0;
    return TPMC_OK;
  }
  if (cfg->bvh_leaf > 127) return fail(TPMC_EINVAL, "bvh_leaf must be in [0, 127]");
  if (cfg->bvh_width != 0 && cfg->bvh_width != 2 && cfg->bvh_width != 4 && cfg->bvh_width != 8)
    return fail(TPMC_EINVAL, "bvh_width must be 0, 2, 4 or 8");
  if (cfg->block == 0) {  // the BVH layout of later loads only
    c->bvh_leaf = cfg->bvh_leaf ? cfg->bvh_leaf : 4;
    c->bvh_width = cfg->bvh_width;
    return TPMC_OK;
  }
  if (cfg->block % 32 != 0 || cfg->block > 256) return fail(TPMC_EINVAL, "block must be 32..256, multiple of 32");
  if (cfg->chunk != 0 && (cfg->chunk % 32 != 0)) return fail(TPMC_EINVAL, "chunk must be a multiple of 32");
  if (cfg->refill_at > 32) return fail(TPMC_EINVAL, "refill_at must be in [0, 32]");
  if (cfg->bvh_leaf > 127) return fail(TPMC_EINVAL, "bvh_leaf must be in [0, 127]");
  c->manual_launch = true;
  c->manual.block = cfg->block;
  c->manual.blocks_per_sm = cfg->blocks_per_sm;
  c->manual.chunk = cfg->chunk;
  c->manual.smem_nodes = cfg->smem_nodes;
  c->manual.refill_at = cfg->refill_at;
  c->bvh_leaf = cfg->bvh_leaf ? cfg->bvh_leaf : 4;
  c->bvh_width = cfg->bvh_width;
  return TPMC_OK;
}

tpmc_status tpmc_get_launch(tpmc_ctx* ctx, tpmc_mesh_id mesh, uint32_t precision, tpmc_launch* out) {
  if (!ctx || !out) return fail(TPMC_EINVAL, "NULL argument");
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  std::lock_guard<std::recursive_mutex> lk(c->mu);
  auto it = c->meshes.find(mesh);
  if (it == c->meshes.end()) return fail(TPMC_ENOTFOUND, "unknown mesh id");
  const LaunchCfg cfg = c->schedule(
      it->second, precision | (it->second.dev.width == 8 ? kVariantWide8 : (it->second.dev.width == 4 ? kVariantWide4 : 0u)), 0);
  out->block = cfg.block;
  out->blocks_per_sm = cfg.blocks_per_sm;
  out->chunk = cfg.chunk;
  out->smem_nodes = cfg.smem_nodes;
  out->refill_at = cfg.refill_at;
  out->bvh_leaf = c->bvh_leaf;
  out->bvh_width = it->second.dev.width;
  return TPMC_OK;
}

}  // extern "C"
