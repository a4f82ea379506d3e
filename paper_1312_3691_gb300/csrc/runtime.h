// Host-side context of the TPMC library (not part of the ABI).
#pragma once

#include <algorithm>
#include <condition_variable>
#include <cstdint>
#include <deque>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "tpmc_internal.h"

namespace tpmc {

extern thread_local std::string g_last_error;
tpmc_status fail(tpmc_status st, const std::string& msg);
tpmc_status cuda_fail(cudaError_t e, const char* where);
tpmc_status validate_params(const tpmc_params* p);

struct MeshRec {
  MeshDev dev;
  void* d_block = nullptr;     // one device allocation holding every mesh array
  size_t bytes = 0;
  double center[3] = {0, 0, 0}, radius = 0, lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  uint32_t depth = 0, leaf_max = 0, n_skipped = 0, n_vert = 0, n_exposed = 0, node_bytes = 64;
  std::vector<double> h_xyz;   // host copy for the control-volume containment check
  std::vector<uint32_t> h_tri;
  int in_use = 0;              // queries in flight on this mesh (serving)
};

struct PanelRec {
  void* d_panel = nullptr;     // [n_tri][3] int64 fixed-point sums
  QueryDev query;              // set-up values needed for the conversion
  tpmc_mesh_id mesh = 0;
  uint32_t n_tri = 0;
};

struct Scratch {
  void* ptr = nullptr;
  size_t cap = 0;
};

// Seeded particles of a launch's batches (Ctx::grow_pool, Ctx::trace_pool), the
// second stream of the launch and where it leaves and rejoins the first.  Freed
// when another allocation needs the room, after `done` (the serving loop, whose
// locks nobody should wait for, does so between its steps: give_back_pools).
struct Pool {
  void* ptr = nullptr;
  size_t cap = 0;
  uint64_t max_batch = 0;
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr, done = nullptr;
};

struct ServeState;  // serve.cpp

// Items of a sweep whose inputs and results stay in the context's pinned memory.
constexpr uint32_t kPinnedItems = 256;
constexpr size_t kPinnedBytes = 256 + kPinnedItems * (sizeof(tpmc_result) + 4 * sizeof(double));

// BVH width of mesh loads that neither tpmc_set_launch nor tpmc_tune decided.
constexpr uint32_t kDefaultBvhWidth = 2;

// FP32 launches of at least this many particles go through the pool.  Below, the
// second launch and two tails cost what the leaner kernels save.  us fused / through
// the pool at S = 7, eps = 0.9: one query of 2^21 and 2^22 particles, then 16 queries
// of 2^20 and 2^22 in all:
//   plate       169/178    277/263     162/161  339/245
//   icosphere   548/513    1013/890    448/377  1362/1023
//   cylinder    337/470    582/558     316/299  829/680
//   hemisphere  1886/1711  3358/3001   875/787  2159/1772
//   satellite   532/518    674/597     761/758  1154/946
// (one query of 2^22 at three S and directions: the cylinder 5 % faster to 2 %
// slower, the other bodies 3 to 21 % faster)
constexpr uint64_t kPoolMin = 1u << 22;
// Particles of a batch, at most and, in a launch of several, at least (32 bytes
// each, two batches).  Every batch has a tail of its own, the fused launch one for
// all.  ms for 1e8 particles of one query and for 96 queries of 1e6, fused, then
// in batches of 2^20, 2^22, 2^23 and 2^26:
//   plate       5.1 4.8    6.5 5.3    4.7 3.7    4.4 3.4    4.2 3.2
//   icosphere   22.6 24.0  21.8 22.8  19.3 20.4  18.4 19.3  18.0 18.6
//   cylinder    12.1 13.6  19.3 16.3  11.7 13.0  10.7 11.3  9.6 10.2
//   hemisphere  71.1 31.2  79.6 40.1  65.8 31.2  63.0 28.2  61.4 27.6
//   satellite   7.3 9.7    23.5 26.8  9.4 11.5   6.9 8.7    5.2 6.2
constexpr uint64_t kPoolBatch = 1ull << 26, kPoolSmallest = 1ull << 23;
// Batches that a call which only enqueues (tpmc_sweep_device, a serving step) puts
// into its two streams, each of which gets as many launches: a stream's queue holds
// about 1,024, and beyond that the host waits for the GPU with the context's lock
// held (2^35 particles in batches of 2^23 on no mesh: 346 of 461 ms; now 4).  What is
// left is one launch.
constexpr uint64_t kPoolBatchesQueued = 896;
constexpr uint32_t kPoolSegment = 2048;  // work indices of a segment, at most (a batch is a multiple)

// Bytes of a pool of `entries` particles (a multiple of 2 kPoolSegment), in two halves: the particles and a count for
// each segment of 32 or more.
constexpr size_t pool_bytes(uint64_t entries) {
  return (size_t)entries * kPoolEntryBytes + (size_t)(entries / 32) * sizeof(uint32_t) + 512;
}

// Particles of a batch in a pool of `entries`: a launch that fits into it, and into
// max_batch, is one batch; others take its two halves in turn.
constexpr uint64_t pool_batch(uint64_t entries, uint64_t total, uint64_t max_batch) {
  return std::min(total <= entries && total <= max_batch ? entries : entries / 2, max_batch);
}

// Entries of a pool for launches of `total` particles that takes at most half of
// `room` bytes; 0: there is no room for one.  Powers of two, so that a program that
// raises its count from call to call does not free and allocate a pool at each (40
// calls of 2^24 particles and 2^20 more at each on a 60,000-triangle satellite: 161
// -> 92 ms, 89 when repeated).  A launch of one batch may be smaller than
// kPoolSmallest, one of several has batches of at least that.
constexpr uint64_t pool_entries(uint64_t total, uint64_t max_batch, size_t room) {
  uint64_t n = 2 * kPoolSegment;
  while (n < total && n < 2 * max_batch) n *= 2;
  while (n > kPoolSegment && pool_bytes(n) > room / 2) n /= 2;
  const bool one = total <= n && total <= max_batch;
  return n > kPoolSegment && (one || n >= 2 * kPoolSmallest) ? n : 0;
}

float cv_area(const QueryDev& q);
tpmc_status fill_query(const MeshRec& m, const tpmc_params* p, uint64_t N, QueryDev* q);

inline uint64_t tune_key(uint32_t n_tri, uint32_t variant) {
  // size classes: powers of 4 of the triangle count; one table per kernel variant
  uint32_t cls = 0;
  while (n_tri > 1 && cls < 16) { n_tri >>= 2; ++cls; }
  return ((uint64_t)variant << 32) | cls;
}

struct Ctx {
  int device = 0;
  int num_sms = 1;
  cudaStream_t own_stream = nullptr;
  cudaStream_t stream = nullptr;
  size_t budget = 0, used = 0;
  uint64_t n_allocs = 0;       // device allocations made since creation
  std::map<void*, size_t> sizes;
  std::recursive_mutex mu;
  std::map<tpmc_mesh_id, MeshRec> meshes;
  tpmc_mesh_id next_mesh = 1;
  std::map<tpmc_query_id, PanelRec> panels;
  tpmc_query_id next_query = 1;
  bool counters = false;
  bool manual_launch = false;
  bool pool_always = false;    // while the tuner times both sizes of a long trial (tune.cpp: measure)
  uint32_t bvh_leaf = 4;       // largest leaf of the BVHs built by later mesh loads
  uint32_t bvh_width = 0;      // children per node of later mesh loads (0: tuned or default)
  std::map<uint64_t, uint32_t> tuned_width;  // BVH width chosen by tpmc_tune per size class
  LaunchCfg manual;
  LaunchCfg last_cfg;
  std::map<uint64_t, LaunchCfg> tuned;
  std::map<uint64_t, int> max_blocks;  // trace_max_blocks_per_sm by variant, block and shared memory
  Scratch s_queries, s_acc, s_items, s_misc, s_out, s_in;
  Pool pool;                   // of the calls on `stream`
  std::vector<Pool*> pools{&pool};  // all of them (the serving steps have their own)
  float* vn_table = nullptr;   // start tables (normal speed, latitude knots), built once at creation
  void* h_pinned = nullptr;
  int* h_err_word = nullptr;          // in h_pinned, as are the next two
  tpmc_result* h_results = nullptr;   // [kPinnedItems], written by the reduction
  double* h_inputs = nullptr;         // [kPinnedItems][4] directions and speed ratios, read by the set-up
  ServeState* serve = nullptr;

  uint32_t width_for(uint32_t n_tri) const;
  tpmc_status upload_mesh(const double* xyz, uint32_t n_vert, const uint32_t* tri, uint32_t n_tri, uint32_t width,
                          MeshRec* out);
  tpmc_status alloc(void** p, size_t bytes, const char* what, bool take_pools = true);
  void release(void* p);
  tpmc_status grow(Scratch& s, size_t bytes, const char* what);
  LaunchCfg schedule(const MeshRec& m, uint32_t variant, uint64_t total);  // variant: see trace_variant
  tpmc_status run(const MeshRec& m, uint32_t nq, const QueryDev& base, const double* d_dirs, const double* d_S,
                  uint64_t total, uint32_t variant, tpmc_result* d_out, const RecordsDev* rec,
                  uint64_t max_batches = ~0ull);
  bool grow_pool(Pool& pool, uint64_t total, uint64_t max_batch);
  void release_pool(Pool& pool);
  bool release_pools();
  size_t pooled() const;
  void destroy_pool(Pool& pool);
  cudaError_t trace_pool(Pool& pool, cudaStream_t stream, TraceArgs a, uint32_t variant, const LaunchCfg& cfg,
                         const MeshRec& m, float area, uint64_t max_batches);
  tpmc_status check_error_word();
  ~Ctx();
};

void stop_serving(Ctx* c);
// Wakes the serving scheduler after device memory was released outside it
// (panel loads read by tpmc_panels), so that queries waiting for memory retry.
void serve_memory_released(Ctx* c);

}  // namespace tpmc
