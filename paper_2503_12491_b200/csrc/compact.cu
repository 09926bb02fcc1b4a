// Gather-compaction of the retained K/V rows into the packed varlen cache
// (Eq. 12: K^ = K[D,:], V^ = V[D,:]) and the position getter.
//
// The survivor lists are in bucket order; the packed cache is in ascending token position.
// Positions are distinct integers below n, so the ordering is a bitmap: every retained
// position sets its bit, and the rank of a bit is the number of bits before it.
#include "cake_internal.cuh"

namespace cake {
namespace {

// First row of every block (r, l) = index r*L + l in the packed cache, and, where asked for, its
// first key group of the 4-bit layout and its first row of the decode cache (one spare row per
// head).  Layers outside [lo, hi) have no rows.  One CTA, block scans over the blocks (one thread
// that walked them took 4 us at 64 blocks, 11 us at 256).
constexpr int OFF_THREADS = 1024;
__global__ void __launch_bounds__(OFF_THREADS)
block_offsets(const int32_t* __restrict__ budget, int64_t* __restrict__ row_off, int64_t* __restrict__ key_off,
              int64_t* __restrict__ dec_off, int nblk, int L, int lo, int hi, int Hkv, int Sw, int group) {
  __shared__ int64_t tot[2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = (int)blockDim.x >> 5;
  int64_t base0 = 0, base1 = 0;                       // rows and key groups (or heads) so far
  for (int i0 = 0; i0 < nblk; i0 += (int)blockDim.x) {
    const int i = i0 + (int)threadIdx.x, l = i % L;
    int64_t a = 0, b = 0;
    if (i < nblk && l >= lo && l < hi) {
      const int len = budget[i] + Sw;
      a = (int64_t)Hkv * len;
      b = key_off ? (int64_t)Hkv * ((len + group - 1) / group) : (int64_t)Hkv;
    }
    int64_t sa = a, sb = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t na = __shfl_up_sync(0xffffffffu, sa, o), nb = __shfl_up_sync(0xffffffffu, sb, o);
      if (lane >= o) { sa += na; sb += nb; }
    }
    if (lane == 31) { tot[0][warp] = sa; tot[1][warp] = sb; }
    __syncthreads();
    int64_t pa = base0, pb = base1;
    for (int w = 0; w < n_warps; ++w) {
      if (w < warp) { pa += tot[0][w]; pb += tot[1][w]; }
      base0 += tot[0][w];
      base1 += tot[1][w];
    }
    pa += sa - a;
    pb += sb - b;
    if (i < nblk) {
      row_off[i] = pa;
      if (key_off) key_off[i] = pb;
      if (dec_off) dec_off[i] = pa + pb;             // a spare row per head
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    row_off[nblk] = base0;
    if (key_off) key_off[nblk] = base1;
    if (dec_off) dec_off[nblk] = base0 + base1;
  }
}

constexpr int kTieCap = 2048;

struct EvictSmem {
  uint32_t hist[1024];
  int32_t ties[kTieCap];
  int warp_tot[32];
  int total;
  uint32_t sel_digit, sel_rem, sel_cnt;
  int32_t tie_count, pos_cut;
};

// Among `cnt` entries (all in one bucket), finds the digit (10 bits at `shift`) that holds the
// krem-th largest key among the entries whose bits above shift+10 equal `prefix_bits`.
__device__ inline void radix_digit(const uint2* __restrict__ e, int cnt, uint32_t mask,
                                   uint32_t prefix_bits, int shift, uint32_t krem, EvictSmem& S) {
  for (int b = threadIdx.x; b < 1024; b += blockDim.x) S.hist[b] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const uint32_t key = __ldcg(&e[i]).x;
    if ((key & mask) == prefix_bits) atomicAdd(&S.hist[(key >> shift) & 1023u], 1u);
  }
  __syncthreads();
  // digits from the top: thread t owns digits 1023-4t .. 1020-4t
  const int per = 1024 / blockDim.x;
  int mine = 0;
  for (int q = 0; q < per; ++q) mine += (int)S.hist[1023 - (threadIdx.x * per + q)];
  int above = block_excl_scan(mine, S.warp_tot, &S.total);
  for (int q = 0; q < per; ++q) {
    const int dg = 1023 - (threadIdx.x * per + q);
    const int h = (int)S.hist[dg];
    if ((uint32_t)above < krem && (uint32_t)(above + h) >= krem) {
      S.sel_digit = (uint32_t)dg;
      S.sel_rem = krem - (uint32_t)above;
      S.sel_cnt = (uint32_t)h;
    }
    above += h;
  }
  __syncthreads();
}

// Where the budget b cuts one list: the retained set is its first b entries in the order (indicator
// descending, position ascending)  (Section 4.2 EVICT, Eq. 12).
__device__ void list_threshold(const int32_t* __restrict__ pf, const uint2* __restrict__ list, int b, ListState* out,
                               EvictSmem& S) {
  if (b <= 0) {
    if (threadIdx.x == 0) *out = ListState{-1, 0xFFFFFFFFu, -1, 0};
    return;
  }
  // threshold bucket d: first bucket with prefix[d+1] >= b
  int less = 0;
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) less += __ldcg(&pf[i + 1]) < b ? 1 : 0;
  block_excl_scan(less, S.warp_tot, &S.total);
  const int d = S.total;
  __syncthreads();
  if (d >= kBins) {                                  // b exceeds the stored entries: keep all
    if (threadIdx.x == 0) *out = ListState{kBins - 1, 0u, 0x7FFFFFFF, __ldcg(&pf[kBins])};
    return;
  }
  const int start = __ldcg(&pf[d]), cnt = __ldcg(&pf[d + 1]) - start;
  const uint32_t rem = (uint32_t)(b - start);
  if ((int)rem >= cnt) {
    if (threadIdx.x == 0) *out = ListState{d, 0u, 0x7FFFFFFF, b};
    return;
  }
  const uint2* e = list + start;
  constexpr int low = 32 - kBinBits;                 // key bits below the bucket bits (20)
  radix_digit(e, cnt, 0u, 0u, low - 10, rem, S);
  uint32_t pre = S.sel_digit << (low - 10);
  uint32_t krem = S.sel_rem;
  __syncthreads();
  radix_digit(e, cnt, 1023u << (low - 10), pre, 0, krem, S);
  pre |= S.sel_digit;
  const uint32_t need_eq = S.sel_rem, n_eq = S.sel_cnt;
  __syncthreads();
  // full key of the threshold: bucket bits + the 20 selected bits
  const uint32_t thr = ((uint32_t)(kBins - 1 - d) << low) | pre;
  int32_t pos_cut = 0x7FFFFFFF;
  if (need_eq < n_eq) {
    // ties at the threshold: the need_eq lowest positions win
    if (threadIdx.x == 0) { S.tie_count = 0; S.pos_cut = 0x7FFFFFFF; }
    __syncthreads();
    if (n_eq <= (uint32_t)kTieCap) {
      for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
        const uint2 v = __ldcg(&e[i]);
        if (v.x == thr) S.ties[atomicAdd(&S.tie_count, 1)] = (int32_t)v.y;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < (int)n_eq; i += blockDim.x) {
        const int32_t p = S.ties[i];
        uint32_t r = 0;
        for (int o = 0; o < (int)n_eq; ++o) r += S.ties[o] < p ? 1u : 0u;
        if (r == need_eq - 1) S.pos_cut = p;
      }
      __syncthreads();
    } else {
      // many ties: bisect the position (positions are distinct)
      int lo = 0, hi = 0x7FFFFFFF;                   // smallest cut with count(pos <= cut) >= need_eq
      while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        int c = 0;
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
          const uint2 v = __ldcg(&e[i]);
          c += (v.x == thr && (int32_t)v.y <= mid) ? 1 : 0;
        }
        block_excl_scan(c, S.warp_tot, &S.total);
        const int tot = S.total;
        __syncthreads();
        if ((uint32_t)tot >= need_eq) hi = mid; else lo = mid + 1;
      }
      if (threadIdx.x == 0) S.pos_cut = lo;
      __syncthreads();
    }
    pos_cut = S.pos_cut;
  }
  if (threadIdx.x == 0) *out = ListState{d, thr, pos_cut, b};
}


// One CTA per (head, layer in [lo, hi), request): where the current budget cuts the list (kept in
// its state for whoever needs the stored indicators too), then the retained positions in ascending order, then the window, written at out[base + g*len ...].  `bitmap` is dynamic
// shared memory when the request's n bits fit, else a slice of global scratch.
template <int POS_THREADS>
__global__ void __launch_bounds__(POS_THREADS)
sorted_positions(const uint2* __restrict__ lists, const int32_t* __restrict__ prefix_all,
                 ListState* __restrict__ states, const ReqInfo* __restrict__ reqs,
                 const int32_t* __restrict__ budget, const int64_t* __restrict__ offsets,
                 int32_t* __restrict__ out, uint32_t* __restrict__ scratch, int64_t scratch_words,
                 int req0, int lo, int L, int Hkv, int Sw, int smem_words, int64_t capacity) {
  extern __shared__ uint32_t sh_bits[];
  __shared__ int warp_tot[32];
  __shared__ EvictSmem S;
  __shared__ ListState st;
  const int g = blockIdx.x, layer = lo + blockIdx.y, req = req0 + blockIdx.z;
  const ReqInfo rq = reqs[req];
  const size_t lid = ((size_t)req * L + layer) * Hkv + g;
  const int b = budget[(size_t)req * L + layer];
  const int len = b + Sw;
  int32_t* dst = out + (offsets ? offsets[(size_t)req * L + layer] : 0) + (int64_t)g * len;
  // without row offsets the caller gave a capacity: never write past it
  const int64_t room = offsets ? (int64_t)len : capacity - (int64_t)g * len;
  const int words = (rq.n + 31) >> 5;
  uint32_t* bits = sh_bits;
  const bool in_smem = words <= smem_words;
  if (!in_smem) {
    const size_t cta = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    bits = scratch + cta * (size_t)scratch_words;
  }
  for (int wi = threadIdx.x; wi < words; wi += POS_THREADS) bits[wi] = 0;
  if (in_smem) __syncthreads(); else { __threadfence_block(); __syncthreads(); }
  const int32_t* pf = prefix_all + lid * (kBins + 1);
  const uint2* list = lists + rq.list_off + ((size_t)layer * Hkv + g) * rq.n;
  // a list never grows again (Proposition 1): entries beyond the budget it arrived with were not stored
  const int arrived = states[lid].kept;
  list_threshold(pf, list, min(min(b, rq.n), arrived), &st, S);
  __syncthreads();
  if (threadIdx.x == 0) states[lid] = ListState{st.bucket, st.thr_key, st.pos_cut, arrived};
  if (st.bucket >= 0 && b > 0) {
    const int start = pf[st.bucket], end = pf[st.bucket + 1];
    for (int i = threadIdx.x; i < end; i += POS_THREADS) {
      const uint2 e = list[i];
      const bool keep = i < start || e.x > st.thr_key || (e.x == st.thr_key && (int32_t)e.y <= st.pos_cut);
      if (keep && e.y < (uint32_t)rq.n) atomicOr(&bits[e.y >> 5], 1u << (e.y & 31));
    }
  }
  __syncthreads();
  // rank of every word, then expand
  const int per = (words + POS_THREADS - 1) / POS_THREADS;
  const int w0 = threadIdx.x * per, w1 = min(words, w0 + per);
  int cnt = 0;
  for (int wi = w0; wi < w1; ++wi) cnt += __popc(bits[wi]);
  // exclusive scan over the block
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < POS_THREADS / 32 ? warp_tot[lane] : 0;
    int winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += n;
    }
    warp_tot[lane] = winc - w;
  }
  __syncthreads();
  int rank = warp_tot[warp] + inc - cnt;
  for (int wi = w0; wi < w1; ++wi) {
    uint32_t m = bits[wi];
    while (m) {
      const int bit = __ffs(m) - 1;
      m &= m - 1;
      if (rank < b && rank < room) dst[rank] = (wi << 5) + bit;
      ++rank;
    }
  }
  for (int t = threadIdx.x; t < Sw; t += POS_THREADS)
    if (b + t < room) dst[b + t] = rq.n + t;
}

constexpr int GA_THREADS = 128;
constexpr int GA_BATCH = 8;                          // passes of K and of V loads a warp has in flight

// Copies the retained rows, one warp per 32 consecutive packed rows: every lane finds the source of
// one row, then the warp copies them CPR lanes (16 bytes each) to a row.  With dec_off the rows go into
// the decode layout, one spare row (written as zero) behind every head's rows.
//
// Bound: memory; rows of 256 bytes at random places.  One lookup (a binary search and a 64-bit division) per
// row and four rows in flight took 210 us for 1.05 M rows of 256 bytes in K and V (5.1 TB/s).
template <int CPR, bool kDecode>
__global__ void __launch_bounds__(GA_THREADS)
gather_rows(const LayerPtrs ptrs, const int64_t* __restrict__ offsets, const int64_t* __restrict__ dec_off,
            const int32_t* __restrict__ budget, const int32_t* __restrict__ pos_packed, const ReqInfo* __restrict__ reqs,
            uint4* __restrict__ k_out, uint4* __restrict__ v_out, int n_req, int L, int Hkv, int Sw, int64_t T) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int RPP = 32 / CPR, NIT = 32 / RPP, NB = NIT < GA_BATCH ? NIT : GA_BATCH;
  const int nblk = n_req * L;
  const int64_t total = offsets[nblk];
  const int lane = threadIdx.x & 31, sub = lane / CPR, chunk = lane % CPR;
  const int64_t n_warps = ((int64_t)gridDim.x * GA_THREADS) >> 5;
  for (int64_t base = (((int64_t)blockIdx.x * GA_THREADS + threadIdx.x) >> 5) * 32; base < total; base += n_warps * 32) {
    // the block of the first row, 32 probes at a time; a lane's own row lies there or shortly after
    int blk = 0, hi = nblk;
    while (hi - blk > 1) {
      const int step = (hi - blk + 31) / 32, at = blk + lane * step;
      const unsigned below = __ballot_sync(kAll, at < hi && offsets[at] <= base);
      blk += (31 - __clz(below)) * step;
      hi = min(hi, blk + step);
    }
    const int64_t row = min(base + lane, total - 1);
    while (offsets[blk + 1] <= row) ++blk;
    const int r = blk / L, l = blk - r * L, len = budget[blk] + Sw;
    const int rel = (int)(row - offsets[blk]), g = rel / len;
    const size_t src = ((size_t)g * T + reqs[r].cu + pos_packed[row]) * CPR;
    const unsigned long long ks = (unsigned long long)(reinterpret_cast<const uint4*>(ptrs.k[l]) + src);
    const unsigned long long vs = (unsigned long long)(reinterpret_cast<const uint4*>(ptrs.v[l]) + src);
    // where the row goes; in the decode layout also whether a spare row follows it
    long long dst = kDecode ? dec_off[blk] + rel + g : row;
    if (kDecode && rel - g * len == len - 1) dst = ~dst;
    const int n_rows = (int)min((int64_t)32, total - base);
#pragma unroll 1
    for (int b = 0; b < NIT && b * RPP < n_rows; b += NB) {
      uint4 kv[NB], vv[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int from = (b + j) * RPP + sub;
        kv[j] = __ldcs(reinterpret_cast<const uint4*>(__shfl_sync(kAll, ks, from)) + chunk);
        vv[j] = __ldcs(reinterpret_cast<const uint4*>(__shfl_sync(kAll, vs, from)) + chunk);
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int from = (b + j) * RPP + sub;
        const long long d = __shfl_sync(kAll, dst, from);
        if (from < n_rows) {
          const size_t o = (size_t)(d < 0 ? ~d : d) * CPR + chunk;
          k_out[o] = kv[j];
          v_out[o] = vv[j];
          if (kDecode && d < 0) k_out[o + CPR] = v_out[o + CPR] = make_uint4(0, 0, 0, 0);
        }
      }
    }
  }
}

}  // namespace

int32_t run_offsets(cake_ctx* ctx, int lo, int hi, int64_t* row_off, int64_t* key_off, int group, int64_t* dec_off,
                    cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int nblk = ctx->n_req * c.n_layers;
  const int threads = nblk >= OFF_THREADS ? OFF_THREADS : nblk > 32 ? (nblk + 31) / 32 * 32 : 32;
  block_offsets<<<1, threads, 0, st>>>(ctx->n_req > 0 ? ctx->d_budget[(ctx->n_evicted - 1) & 1] : nullptr, row_off, key_off,
                                       dec_off, nblk, c.n_layers, lo, hi, c.n_kv_heads, c.window, group);
  count_launch();
  return cuda_status(cudaGetLastError());
}

int32_t run_sorted_positions(cake_ctx* ctx, int req0, int n_req, int lo, int hi, const int64_t* offsets,
                             int32_t* out, int64_t capacity, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  if (n_req <= 0 || hi <= lo) return CAKE_OK;
  const int32_t* budget = ctx->d_budget[(ctx->n_evicted - 1) & 1];
  int max_n = 0;
  for (int r = req0; r < req0 + n_req; ++r) max_n = ctx->h_req[r].n > max_n ? ctx->h_req[r].n : max_n;
  int need_words = (max_n + 31) / 32;
  int smem_words = need_words < kBitmapSmemWords ? need_words : kBitmapSmemWords;
  static PerDeviceOnce attr;
  if (attr.need(ctx->device)) {
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitmapSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitmapSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitmapSmemWords * 4));
    attr.mark(ctx->device);
  }
  const int64_t ctas = (int64_t)c.n_kv_heads * (hi - lo) * n_req;
  if (need_words > kBitmapSmemWords &&
      (!ctx->d_bitmap || ctas * (int64_t)need_words > ctx->bitmap_words)) return CAKE_ERR_CAPACITY;
  const dim3 grid(c.n_kv_heads, hi - lo, n_req);
  // A list is a chain of scans and short passes: with more lists than the device holds CTAs of 1024
  // threads, smaller ones keep more chains in flight (1024 lists of 4K tokens: 42 us with 1024 threads).
#define CAKE_POSITIONS(NT)                                                                                                \
  sorted_positions<NT><<<grid, NT, (size_t)smem_words * 4, st>>>(                                                         \
      ctx->d_lists, ctx->d_prefix, ctx->d_lstate, ctx->d_req, budget, offsets, out, ctx->d_bitmap, need_words, req0, lo,  \
      c.n_layers, c.n_kv_heads, c.window, smem_words, capacity)
  if (ctas <= 2 * ctx->n_sm) CAKE_POSITIONS(1024);
  else if (ctas <= 4 * ctx->n_sm) CAKE_POSITIONS(512);
  else CAKE_POSITIONS(256);
#undef CAKE_POSITIONS
  count_launch();
  return cuda_status(cudaGetLastError());
}

// Rows of the packed order into k_out / v_out (dec_off: into the decode layout).
int32_t run_gather(cake_ctx* ctx, const LayerPtrs& ptrs, const int64_t* row_off, const int64_t* dec_off, const int32_t* pos,
                   void* k_out, void* v_out, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int32_t* budget = ctx->d_budget[(ctx->n_evicted - 1) & 1];
  const int grid = ctx->n_sm * 5;
#define CAKE_GATHER(CPR)                                                                                                 \
  if (dec_off)                                                                                                           \
    gather_rows<CPR, true><<<grid, GA_THREADS, 0, st>>>(ptrs, row_off, dec_off, budget, pos, ctx->d_req, (uint4*)k_out,  \
                                                        (uint4*)v_out, ctx->n_req, c.n_layers, c.n_kv_heads, c.window,   \
                                                        ctx->total_tokens);                                              \
  else                                                                                                                   \
    gather_rows<CPR, false><<<grid, GA_THREADS, 0, st>>>(ptrs, row_off, dec_off, budget, pos, ctx->d_req, (uint4*)k_out, \
                                                         (uint4*)v_out, ctx->n_req, c.n_layers, c.n_kv_heads, c.window,  \
                                                         ctx->total_tokens)
  switch (c.head_dim * (c.dtype == CAKE_DTYPE_FP32 ? 4 : 2) / 16) {
    case 8: CAKE_GATHER(8); break;
    case 16: CAKE_GATHER(16); break;
    default: CAKE_GATHER(32); break;
  }
#undef CAKE_GATHER
  count_launch();
  return cuda_status(cudaGetLastError());
}

int32_t launch_compact(cake_ctx* ctx, int32_t lo, int32_t hi, const LayerPtrs& ptrs, void* k_out,
                       void* v_out, int64_t* row_offsets, int32_t* positions, cudaStream_t st) {
  int32_t rc = run_offsets(ctx, lo, hi, row_offsets, nullptr, 1, nullptr, st);
  if (rc != CAKE_OK || ctx->n_req == 0 || hi <= lo) return rc;
  // positions in packed row order: into the caller's buffer if there is one
  int32_t* pos = positions ? positions : ctx->d_pos_packed;
  rc = run_sorted_positions(ctx, 0, ctx->n_req, lo, hi, row_offsets, pos, 0, st);
  if (rc != CAKE_OK) return rc;
  return run_gather(ctx, ptrs, row_offsets, nullptr, pos, k_out, v_out, st);
}

int32_t launch_get_positions(cake_ctx* ctx, int32_t req, int32_t layer, int32_t* out,
                             int64_t capacity, cudaStream_t st) {
  if (capacity < 0) return CAKE_ERR_ARG;
  return run_sorted_positions(ctx, req, 1, layer, layer + 1, nullptr, out, capacity, st);
}

namespace {
struct ClearArgs {
  uint8_t* buf[CAKE_CLEAR_MAX];
  const int64_t* used[CAKE_CLEAR_MAX];
  int64_t row_bytes[CAKE_CLEAR_MAX], rows[CAKE_CLEAR_MAX];
};
// Rows [*used, rows) of every buffer; blockIdx.y = buffer.  Usually a few rows or none.
__global__ void clear_unused(const ClearArgs A) {
  const int b = blockIdx.y;
  const int64_t lo = *A.used[b] * A.row_bytes[b], hi = A.rows[b] * A.row_bytes[b];
  uint8_t* p = A.buf[b];
  const int64_t mid = min(hi, (lo + 15) & ~(int64_t)15), last = max(mid, hi & ~(int64_t)15);   // 16-byte part, if aligned
  const bool vec = ((uintptr_t)p & 15) == 0;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  if (vec) {
    for (int64_t i = lo + t; i < mid; i += nt) p[i] = 0;
    for (int64_t i = mid / 16 + t; i < last / 16; i += nt) reinterpret_cast<uint4*>(p)[i] = make_uint4(0, 0, 0, 0);
    for (int64_t i = last + t; i < hi; i += nt) p[i] = 0;
  } else {
    for (int64_t i = lo + t; i < hi; i += nt) p[i] = 0;
  }
}
}  // namespace

}  // namespace cake

extern "C" int32_t cake_clear_unused(int32_t n, void* const* bufs, const int64_t* row_bytes, const int64_t* rows,
                                     const int64_t* const* used_rows, void* stream) {
  using namespace cake;
  if (n < 0 || n > CAKE_CLEAR_MAX || (n > 0 && (!bufs || !row_bytes || !rows || !used_rows))) return CAKE_ERR_ARG;
  if (n == 0) return CAKE_OK;
  ClearArgs A;
  for (int i = 0; i < n; ++i) {
    if (!bufs[i] || !used_rows[i] || row_bytes[i] < 0 || rows[i] < 0) return CAKE_ERR_ARG;
    A.buf[i] = (uint8_t*)bufs[i];
    A.used[i] = used_rows[i];
    A.row_bytes[i] = row_bytes[i];
    A.rows[i] = rows[i];
  }
  clear_unused<<<dim3(64, n), 256, 0, (cudaStream_t)stream>>>(A);
  count_launch();
  return cuda_status(cudaGetLastError());
}
