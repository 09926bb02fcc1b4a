// Internal declarations shared by the translation units of libcake.
#pragma once

#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cuda_bf16.h>
#include <stdint.h>

#include "cake.h"

namespace cake {

constexpr int kMaxRows = 128;        // G * S_w rows handled per KV head
constexpr int kSimtMinUnit = 64;      // fewest keys of a score unit of the SIMT score kernels
constexpr int kSimtMaxUnit = 1024;
constexpr int64_t kMaxScoreElems = 64ll << 20;   // logits the SIMT kernels keep between their two steps (256 MB)
constexpr int kSimtThreads = 256;
constexpr int kBins = 4096;          // buckets of the indicators, see bucket_of
constexpr int kChunkKeys = 4096;     // granularity of the token ranges of the pooling
constexpr int kBitmapSmemWords = 36 * 1024;   // positions of up to 1.1 M tokens are ordered in a CTA's shared memory
constexpr int kSelectSmemWords = 50 * 1024;   // dynamic shared memory of the selection: queues, bitmap and list of candidates
constexpr int kScoreDepth = 8;        // layers whose score outputs may wait for their pooling, where memory allows
constexpr int kScoreGroups = 3;      // statistics warp groups per CTA of the tensor-core score kernel
constexpr int kScoreWarps = 4 * kScoreGroups;   // statistics warps: one column-pass partial each

// One request of the current batch (device copy in ctx->d_req).
struct ReqInfo {
  int64_t cu;        // first token row of the request inside the packed K/V
  int32_t N;         // prompt length
  int32_t n;         // N - S_w non-window tokens
  int32_t keep_all;  // 1: N <= floor(B_total/L), nothing is evicted
  int32_t pad;
  int32_t unit0;     // first score unit of the request
  int32_t nunits;    // number of score units of the request
};

// A run of consecutive keys of one request handled by one CTA of a score kernel.
struct ScoreUnit {
  int64_t cu;        // first token row of the request inside the packed K
  int32_t req;
  int32_t key0;
  int32_t nkeys;
  int32_t n;         // non-window keys of the request
  int32_t unit0;     // first unit of the request
  int32_t nunits;    // units of the request
};

// One step of a CTA's program in the tensor-core score kernel: a run of consecutive
// keys of one (request, KV head) in pass A (phase 0, row statistics) or pass B (phase 1,
// column statistics).  `seg` numbers the partial results the step writes (one per
// statistics warp group).
struct ScoreOp {
  int64_t base;    // row of the pair's first key in the packed K: g * T + cu[req]
  int32_t req;
  int32_t g;
  int32_t key0;
  int32_t nkeys;
  int32_t phase;
  int32_t seg;
  int32_t n;       // non-window keys of the request
};

// Where a call was enqueued: the stream, by its unique id or in a capture by its handle (0:
// unknown), and the stream capture that recorded it (0: none, the step ran).
struct StepPlace {
  unsigned long long stream, capture;
};
// A read of a budget buffer on a caller's stream that the next write of the buffer has to wait for.
struct BudgetRead {
  cudaEvent_t done;
  bool pending;
  StepPlace at;
};

struct LayerPtrs {
  const void* k[CAKE_MAX_LAYERS];
  const void* v[CAKE_MAX_LAYERS];
};

}  // namespace cake

namespace cake {
struct ProfSpan { int kind; cudaEvent_t a, b; };
struct Profiler {
  bool on;
  int used, cap;
  ProfSpan* spans;
};
}  // namespace cake

struct cake_ctx {
  cake_config cfg;
  cake::Profiler prof;
  int device;
  int n_sm;
  int n_sm_score;          // SMs the persistent score kernel occupies; the rest stay free for the
                           // cascade kernels of the previous layer, which run beside it
  // What follows the scores of layer l (pooling, preference, budgets) runs on an internal stream
  // while the caller's stream already scores layer l+1; events order the two.
  cudaStream_t pool_st;             // pooling, preference and budgets
  cudaEvent_t ev_main, ev_pool_side;   // scratch events: caller's stream -> pool_st, and back
  int32_t score_depth;              // places for score outputs: kScoreDepth, or fewer (see cake_create); layer l uses
                                    // place l % score_depth
  cudaEvent_t ev_score[cake::kScoreDepth];   // score kernel of layer % kScoreDepth has finished
  cudaEvent_t ev_pool[cake::kScoreDepth];    // pooling (the last reader of the score outputs) and budgets of
                                             // layer % kScoreDepth have finished
  bool pool_recorded[cake::kScoreDepth];
  int32_t pool_waited;              // newest layer whose pooling the stream of the latest score launch has waited for
  unsigned long long score_stream;  // that stream (0: unknown)
  int32_t rows;            // R = G * S_w
  int64_t sel_budget;      // B' = B_total - L * S_w
  // ---- batch state (host) ----
  int32_t n_req;
  int64_t total_tokens;    // T
  int32_t n_units;         // score units for all N keys (phase A)
  int32_t n_ind;           // layers whose indicators have arrived
  int32_t n_pref;          // layers whose preference is known
  int32_t n_evicted;       // stages completed
  int32_t alloc_of_buf[2]; // stage whose budgets live in budget buffer 0/1 (-1 none)
  cake::BudgetRead budget_read[2];   // newest read of either buffer on a caller's stream
  int32_t last_alloc;      // most recent stage passed to cake_allocate
  int32_t arrived_budgets; // stage whose budgets were computed when its layer was scored (-1: none, or a
                           // preference was set since)
  int32_t max_n_tokens;    // longest prompt of the batch
  int32_t n_fin_parts;     // teams that share the preference of a request
  int64_t packed_rows_bound;
  int64_t* h_cu;           // host copy of cu_seqlens [max_requests+1]
  // ---- pinned staging ----
  cake::ReqInfo* h_req;    // [max_requests]
  cake::ScoreUnit* h_units;
  cudaEvent_t upload_done;
  bool upload_pending;
  // ---- device state ----
  cake::ReqInfo* d_req;
  cake::ScoreUnit* d_units;
  int32_t max_units;
  double* d_H;             // [max_requests][L]
  double* d_V;
  double* d_P;
  int32_t* d_budget[2];    // [max_requests][L] selectable budgets, double-buffered by stage parity
  int32_t* d_status;       // sticky device status word
  uint8_t* d_ring;         // one allocation for the places of d_raw, d_colpart and d_hrow
  float* d_raw[cake::kScoreDepth];     // [H_kv][max_total_tokens] un-pooled indicator, by layer % score_depth
  float* d_store;          // [L][H_kv][tokens of the batch] pooled indicators of every layer, +inf on the windows
  uint16_t* d_codes;       // [L][H_kv][code_tokens(n_req)] upper half of every indicator's ordered key, see code_row
  int64_t max_lists;       // (request, layer, head) triples
  int32_t* d_prefix;       // [max_lists][kBins+1] bucket offsets of every (request, layer, head)
  uint32_t* d_hist;        // [max_pairs][kBins] bucket histogram of the arriving layer (zero at rest)
  uint32_t* d_arrivals;    // zero at rest: [max_pairs] a list's finished runs in the pooling, [max_requests] a
                           // request's finished parts of the preference
  double* d_headsum;       // [max_requests][H_q][2] per-head entropy / variance sums of the layer
  int32_t* d_pos_packed;   // [packed rows bound] positions in packed row order
  int64_t pos_packed_cap;
  uint32_t* d_bitmap;      // global bitmaps for requests too long for shared memory (or null)
  int64_t bitmap_words;
  float* d_lse2;           // [max_requests][H_q][S_w] base-2 log-sum-exp of window rows
  float2* d_rowpart;       // [max_units][H_kv][R] (max, sum) partials of phase A
  float* d_scores;         // SIMT path: logits between its two kernels
  int64_t scores_elems;
  uint32_t* d_simt_arrivals;   // [max_pairs] finished units of a (request, head) (zero at rest)
  int32_t unit_keys;       // keys of a full score unit of the batch
  float* d_colpart[cake::kScoreDepth]; // partial (sum p*log2 p, sum var) of the column pass, likewise
  // ---- tensor-core score path ----
  bool use_tc;
  bool hhead_from_rows;    // entropy came from pass A (d_hrow) rather than from pass B partials
  int32_t n_tc_ctas, max_tc_segs, max_pairs;
  int32_t n_tc_waves;             // waves of the current plan
  // ---- decode-time eviction (frozen budgets) ----
  bool dec_ready;                 // cake_decode_begin has built the decode state of this batch
  int32_t dec_update_mode;        // CAKE_DECODE_*
  int64_t dec_max_cap;            // slots of the largest head of the batch (len + 1)
  int64_t dec_rows_cap;           // capacity of the three arrays below
  int64_t* d_dec_off;             // [max_requests*L + 1] decode row offsets
  int64_t* d_dec_packed_off;      // [max_requests*L + 1] packed row offsets (set-up scratch)
  float* d_dec_score;             // stored eviction score of every slot
  float* d_dec_tmp;               // [H_kv][tokens + requests][G + 1]: work area of decode heads too large for shared memory
  int32_t* d_dec_pos;             // token position of every slot (-1: free)
  int32_t* d_dec_order;           // per head: rank in ascending position -> slot
  int4* d_dec_meta;               // [max_lists] (len, free slot, next position, frozen budget)
  int32_t* h_budget_stage;        // pinned [max_requests*L] read-back of the final budgets
  int32_t dec_last_layer;         // layer of the latest decode step if it was on the cluster form, else -1
  cake::StepPlace dec_last;       // where that step was enqueued
  cake::StepPlace dec_place[CAKE_MAX_LAYERS];   // the same of every layer's latest step (or of the set-up of the cache)
  bool dec_captured;              // a step of this cache was recorded by a stream capture
  int32_t h_dec_cap[CAKE_MAX_LAYERS];   // slots of the largest head of every layer
  int64_t wait_limit_cycles;      // bound of every device-side wait (0 = the default, about 2 s)
  int32_t debug_epoch_skew;       // test hook: added to the launch count the cross-CTA waits expect
  int32_t n_tc_asegs, n_tc_bsegs;          // pass-A / pass-B segments per layer
  int32_t n_tc_ops_full, n_tc_ops_b, max_tc_ops;
  uint32_t tc_tag;                // both-pass launches since cake_begin: mark of the rows they exchange
  cake::ScoreOp* h_tc_ops;        // pinned: [both-pass programs][pass-B-only programs]
  cake::ScoreOp* d_tc_ops;
  // pinned / device index block of the current batch, P = n_req * H_kv pairs:
  //   pair_aseg [P+1] | pair_bseg [P+1] | group_begin [P+1] | cta_op of the both-pass programs [n_sm+1]
  //   | cta_op of the pass-B-only programs [n_sm+1]
  int32_t n_tc_groups;            // groups of pairs the merger warps take at once
  int32_t* h_tc_index;
  int32_t* d_tc_index;
  int tc_merge_ways;              // rows the merger warp handles side by side (a power of two up to 32), chosen with the plan
  bool tc_direct;                 // every CTA merges the denominators of its own pass-B ops (single-wave plans)
  uint8_t* d_tc_exch;             // rows that the CTAs of a score launch exchange (tc_exchange_bytes); cleared in cake_begin
  float* d_hrow[cake::kScoreDepth];   // [max_pairs][128] sum_j p log2 p per window row, by layer % score_depth
};

namespace cake {

void count_launch(int64_t n = 1);
StepPlace step_place(cudaStream_t st);

// score_simt.cu
int32_t simt_tile_keys(int rows);     // keys per tile: score units are multiples of it
int32_t launch_score_simt(cake_ctx* ctx, int32_t layer, const void* q_win, const void* k,
                          const float* lse, cudaStream_t st);
// score_tc.cu
bool tc_path_supported(const cake_config& c);
size_t tc_index_size(int64_t pairs, int n_sm);
size_t tc_exchange_bytes(int64_t pairs, int64_t segs);
int64_t tc_max_segments(const cake_config& c, int n_sm);
int32_t tc_build_plan(cake_ctx* ctx, int32_t n_req);
int32_t tc_plan_check(const cake_config& c, int n_sm, int reserved, int32_t n_req, const int64_t* cu,
                      int32_t* info8);
int32_t launch_score_tc(cake_ctx* ctx, int32_t layer, const void* q_win, const void* k,
                        const float* lse, cudaStream_t st);
// cascade.cu
int32_t launch_arrive(cake_ctx* ctx, int32_t layer, bool do_pool, bool finalize, bool budgets, cudaStream_t st);
int32_t launch_allocate(cake_ctx* ctx, int32_t stage, cudaStream_t st);
// decode.cu
int32_t launch_decode_begin(cake_ctx* ctx, const LayerPtrs& ptrs, void* k_cache, void* v_cache,
                            int64_t* row_offsets, cudaStream_t st);
int32_t launch_decode_step(cake_ctx* ctx, int32_t layer, const void* q_new, const void* k_new,
                           const void* v_new, void* k_cache, void* v_cache, cudaStream_t st);
int32_t launch_decode_read(cake_ctx* ctx, int32_t req, int32_t layer, int32_t* positions, float* scores,
                           int32_t* slots, cudaStream_t st);
// quant.cu
int32_t launch_compact_int4(cake_ctx* ctx, int32_t lo, int32_t hi, const LayerPtrs& ptrs, int32_t group,
                            uint8_t* k_codes, float* k_scale, float* k_zero, uint8_t* v_codes,
                            float* v_scale, float* v_zero, int64_t* row_offsets, int64_t* kgroup_offsets,
                            int32_t* positions, cudaStream_t st);
// compact.cu
int32_t launch_compact(cake_ctx* ctx, int32_t lo, int32_t hi, const LayerPtrs& ptrs, void* k_out,
                       void* v_out, int64_t* row_offsets, int32_t* positions, cudaStream_t st);
int32_t run_offsets(cake_ctx* ctx, int lo, int hi, int64_t* row_off, int64_t* key_off, int group, int64_t* dec_off,
                    cudaStream_t st);
int32_t run_gather(cake_ctx* ctx, const LayerPtrs& ptrs, const int64_t* row_off, const int64_t* dec_off, const int32_t* pos,
                   void* k_out, void* v_out, cudaStream_t st);
int32_t run_sorted_positions(cake_ctx* ctx, int req0, int n_req, int lo, int hi, const int64_t* offsets,
                             int32_t* out, int64_t capacity, cudaStream_t st);
int32_t launch_get_positions(cake_ctx* ctx, int32_t req, int32_t layer, int32_t* out,
                             int64_t capacity, cudaStream_t st);

// Pooled indicators of a layer of the current batch: [H_kv][T].
inline float* layer_store(const cake_ctx* ctx, int32_t layer) {
  return ctx->d_store + (size_t)layer * ctx->cfg.n_kv_heads * ctx->total_tokens;
}

// Codes of a layer of the current batch: a request's start on a multiple of eight, so that they are written and read in
// vectors whatever the prompts' lengths.
__host__ __device__ inline int64_t code_row(int64_t cu, int64_t r) { return (cu & ~(int64_t)7) + 8 * r; }
inline int64_t code_tokens(int64_t tokens, int64_t n_req) { return code_row(tokens, n_req) + 8; }
inline uint16_t* layer_codes(const cake_ctx* ctx, int32_t layer) {
  return ctx->d_codes + (size_t)layer * ctx->cfg.n_kv_heads * code_tokens(ctx->total_tokens, ctx->n_req);
}

// Global scratch of the selection, for requests whose bitmap does not fit shared memory: words of a (layer, KV head)'s
// bitmaps before request r of a batch, which starts at token cu.  A request of N tokens needs at most
// (N - 1 + 31) / 32 <= N / 32 + 1 words, so that any requests fit between their neighbours.
__host__ __device__ inline int64_t bitmap_words_before(int64_t cu, int64_t r) { return cu / 32 + r; }

// Order-preserving integer image of a float; -0 and +0 compare equal, as they do as floats.
__device__ __forceinline__ uint32_t ordered_key(float v) {
  uint32_t b = __float_as_uint(v);
  b = b == 0x80000000u ? 0u : b;
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}

// A key's bucket, counted from the top (bucket 0 holds the largest values): four to a power of two, and 64 to one between
// 2^-27 and 2^5, where the indicators of prompts of up to millions of tokens lie.  (There every 17th bucket is empty.)
constexpr uint32_t kFineFirst = 0x80000000u | (127u - 27u) << 23, kFineEnd = kFineFirst + (32u << 23);
static_assert((0xFFFFFFFFu >> 21) + ((kFineEnd - kFineFirst) >> 17) == kBins - 1, "every key has a bucket");
__device__ __forceinline__ int bucket_of(uint32_t key) {
  return (int)((kBins - 1) + (kFineFirst >> 17)) - (int)(key >> 21) - (int)(min(max(key, kFineFirst), kFineEnd) >> 17);
}
// (0 beyond the last key: its predecessor ends the topmost buckets)
__device__ __forceinline__ uint32_t bucket_first_key(int bucket) {
  const int bin = kBins - 1 - bucket, fine = bin - (int)(kFineFirst >> 21), steps = (int)((kFineEnd - kFineFirst) >> 17);
  if (fine < 0) return (uint32_t)bin << 21;
  if (fine >= steps + steps / 16) return bin - steps > 2047 ? 0u : (uint32_t)(bin - steps) << 21;
  const int sixteen = fine / 17;
  return kFineFirst + (uint32_t)(16 * sixteen + min(fine - 17 * sixteen, 16)) * (1u << 17);
}
__device__ __forceinline__ uint32_t bucket_last_key(int bucket) { return bucket > 0 ? bucket_first_key(bucket - 1) - 1u : 0xFFFFFFFFu; }

__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// ---- clusters: the rank, barriers, and what a peer has at the place of `p` in its shared memory
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t ld_peer(const void* p, uint32_t rank) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ uint2 ld_peer2(const void* p, uint32_t rank) {
  uint2 v;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(peer_addr(p, rank)) : "memory");
  return v;
}

// The eviction indicator of one key from the mean and variance of its window attention
// (Section 4.3, Eq. 11, and the combinations of the paper's indicator ablation).
__device__ __forceinline__ float combine_indicator(int mode, float gamma, float mean, float var,
                                                   float sw) {
  return mode == CAKE_IND_MEAN_PLUS_VAR ? fmaf(gamma, var, mean)
         : mode == CAKE_IND_MEAN        ? mean
         : mode == CAKE_IND_VAR         ? var
         : mode == CAKE_IND_WINDOW_SUM  ? mean * sw
                                        : mean * var;
}

// Exclusive block scan (blockDim.x <= 1024) of one int per thread; *total gets the sum.
__device__ inline int block_excl_scan(int v, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < nw ? warp_tot[lane] : 0;
    int winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += n;
    }
    warp_tot[lane] = winc - w;
    if (lane == 31) *total = winc;
  }
  __syncthreads();
  const int r = warp_tot[warp] + inc - v;
  __syncthreads();
  return r;
}

// Function attributes (the dynamic shared-memory limit) belong to a device: a flag per device,
// so that a context on a second GPU sets them there too.
constexpr int kOnceDevices = 64;
struct PerDeviceOnce {
  bool done[kOnceDevices] = {};
  bool need(int device) const { return device < 0 || device >= kOnceDevices || !done[device]; }
  void mark(int device) { if (device >= 0 && device < kOnceDevices) done[device] = true; }
};

// The widest cluster a kernel may be launched with: `wide`, beyond the portable 8, only where the current
// device can hold one such cluster of its largest CTAs (a partition of a device, or a share of its SMs, may
// not, and the launch would fail), and never above CAKE_MAX_CLUSTER (environment).  `wide_fits` is what
// cluster_fits said; it allows the kernel such clusters, and answers no where the device cannot say.
template <typename Kernel>
bool cluster_fits(Kernel kernel, int size, int threads, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)size, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)size;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess && n >= 1;
}
constexpr int kPortableCluster = 8;
inline int widest_cluster(bool wide_fits, int wide) {
  const char* env = getenv("CAKE_MAX_CLUSTER");
  const int most = env && env[0] ? atoi(env) : wide;
  const int w = wide_fits ? wide : kPortableCluster;
  return most < 1 ? 1 : most < w ? most : w;
}

// Tracing spans (no-ops unless cake_profile_enable was called).
int prof_begin(cake_ctx* ctx, int kind, cudaStream_t st);
void prof_end(cake_ctx* ctx, int span, cudaStream_t st);

// Maps a CUDA runtime result to a library status; with CAKE_VERBOSE set in the environment the
// runtime's own message goes to stderr, since the status code alone does not say which error it was.
inline int32_t cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return CAKE_OK;
  if (getenv("CAKE_VERBOSE")) fprintf(stderr, "libcake: CUDA error %d: %s\n", (int)e, cudaGetErrorString(e));
  return CAKE_ERR_CUDA;
}

#define CAKE_CUDA_TRY(expr)                         \
  do {                                              \
    cudaError_t _e = (expr);                        \
    if (_e != cudaSuccess) return cuda_status(_e);  \
  } while (0)

}  // namespace cake
