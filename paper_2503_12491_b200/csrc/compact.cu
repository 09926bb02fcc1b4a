// Gather-compaction of the retained K/V rows into the packed varlen cache
// (Eq. 12: K^ = K[D,:], V^ = V[D,:]) and the position getter.
//
// The retained set of a (request, layer, KV head) at a budget b is the first b of its stored indicators in the
// order (indicator descending, position ascending)  (Section 4.2 EVICT, Eq. 12).  It is found here, where it is
// read out, from the indicators and their bucket offsets.  The packed cache is in ascending token position: every retained position sets its bit in a bitmap,
// and the rank of a bit is the number of bits before it.
#include "cake_internal.cuh"

#include <algorithm>

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
  // sorted_positions starts beside this kernel: it waits for it only before it writes
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
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

constexpr int kTieCap = 512;                         // entries of equal rank but for their position that are ranked one by one
constexpr int kFewEntries = 64;                      // entries that are ranked without another histogram
constexpr int SP_BINS = 1024;                        // (22 - clz in the code is 32 - clz - log2 of this)
constexpr int SP_BATCH = 4;                          // groups of 32 entries a warp has in flight

struct SelectSmem {
  uint32_t hist[SP_BINS];
  uint2 ties[kTieCap];                               // (key, position)
  int warp_tot[32];
  int total, count, tie_count;
  int bucket, start, n_in;
  uint32_t sel_bin, sel_rem, sel_cnt;
};

// Bins of the histogram from the top: the one that holds the krem-th entry, how many of its entries are wanted,
// and its size.
__device__ inline void find_bin(uint32_t krem, SelectSmem& S) {
  const int per = max(1, SP_BINS / (int)blockDim.x);
  int mine = 0;
  for (int q = 0; q < per; ++q) mine += (int)S.hist[SP_BINS - 1 - (threadIdx.x * per + q)];
  int above = block_excl_scan(mine, S.warp_tot, &S.total);
  for (int q = 0; q < per; ++q) {
    const int bin = SP_BINS - 1 - (threadIdx.x * per + q), h = (int)S.hist[bin];
    if ((uint32_t)above < krem && (uint32_t)(above + h) >= krem) {
      S.sel_bin = (uint32_t)bin;
      S.sel_rem = krem - (uint32_t)above;
      S.sel_cnt = (uint32_t)h;
    }
    above += h;
  }
  __syncthreads();
}
__device__ inline void clear_hist(SelectSmem& S) {
  for (int i = threadIdx.x; i < SP_BINS; i += blockDim.x) S.hist[i] = 0;
  __syncthreads();
}
// Counts a bin for every lane that has one (>= 0).  Pooled values repeat: a run of equal bins in
// neighbouring lanes is counted once.  Called by whole warps.
__device__ __forceinline__ void count_bin(int bin, SelectSmem& S) {
  if (!__any_sync(0xffffffffu, bin >= 0)) return;
  const int lane = threadIdx.x & 31, before = __shfl_up_sync(0xffffffffu, bin, 1);
  const bool first = lane == 0 || bin != before;
  const uint32_t firsts = __ballot_sync(0xffffffffu, first);
  if (first && bin >= 0) {
    const uint32_t later = lane < 31 ? firsts >> (lane + 1) : 0u;
    atomicAdd(&S.hist[bin], later ? (uint32_t)__ffs(later) : 32u - lane);
  }
}

// One CTA per (head, layer in [lo, hi), request): which positions the current budget b keeps, then these in ascending
// order, then the window, written at out[base + g*len ...].
//   1. The bucket offsets say which bucket holds the b-th largest value, and how many of its entries are wanted.
//   2. One pass over the values, eight to a lane: the bits of those in the buckets before are set, those inside go
//      to a list in shared memory, as (key, position).  If there are too many for it, the steps below go over all values.
//   3. Histograms of SP_BINS equal parts of the bucket's keys narrow it to the bin that holds the b-th value, until that
//      has few entries (usually at once); these are ranked by (key, position).
//   4. Ranks of the bits, positions.
// Bound: the pass over the values, and between the steps the latency of the chain, which other lists' CTAs on the SM
// hide: 46 us for 256 lists of 131 040 values (134 MB), 29 for 512 of 26 000, 20 for 1024 of 4064.  Placing every layer's
// values in bucket order when it arrived made this step 31, 27 and 22 us, for a launch of 7 to 76 us per layer.
// Without the bucket offsets three digit histograms of all values took 300 us in the first case and 137 in the
// second (run lengths, and atomics on few hot bins), and a sample in their place 129 and 133, since the candidates
// on either side of the cut are many where a layer keeps much.  `bits` is shared memory when the request's n
// bits fit, else a slice of global scratch.
template <int POS_THREADS>
__global__ void __launch_bounds__(POS_THREADS, 1024 / POS_THREADS)
sorted_positions(const float* __restrict__ store, const int32_t* __restrict__ prefix_all, const ReqInfo* __restrict__ reqs, const int32_t* __restrict__ budget,
                 const int64_t* __restrict__ offsets, int32_t* __restrict__ out, uint32_t* __restrict__ scratch,
                 int req0, int lo, int L, int Hkv, int Sw, int smem_words, int cap, int64_t T,
                 int64_t capacity) {
  extern __shared__ __align__(16) uint32_t sh_dyn[];
  __shared__ SelectSmem S;
  const int g = blockIdx.x, layer = lo + blockIdx.y, req = req0 + blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int WARPS = POS_THREADS / 32;
  const ReqInfo rq = reqs[req];
  const int n = rq.n;
  const int b = budget[(size_t)req * L + layer];
  const int len = b + Sw;
  // without row offsets the caller gave a capacity: never write past it
  const int64_t room = offsets ? (int64_t)len : capacity - (int64_t)g * len;
  // The offsets are written by the kernel before this one, which may still run; nothing else that is read here is.
  auto row_start = [&]() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the gather waits for this kernel's end
    return out + (offsets ? __ldcg(&offsets[(size_t)req * L + layer]) : 0) + (int64_t)g * len;
  };
  if (b <= 0 || b >= n) {
    int32_t* dst = row_start();
    for (int t = threadIdx.x; t < (b <= 0 ? 0 : n); t += POS_THREADS)
      if (t < room) dst[t] = t;
    for (int t = threadIdx.x; t < Sw; t += POS_THREADS)
      if (b + t < room) dst[b + t] = n + t;
    return;
  }
  // Element q = a + i of the row, counted from the 16-byte boundary at or before its start, is value i: lanes load
  // whole groups of four, and bits and positions count in elements until they are written out.
  const float* const v = store + ((size_t)layer * Hkv + g) * T + rq.cu;
  const int a = (int)((reinterpret_cast<uintptr_t>(v) >> 2) & 3), end = a + n;
  const int words = (end + 31) >> 5;
  uint2* const list = reinterpret_cast<uint2*>(sh_dyn + smem_words);
  uint32_t* bits = sh_dyn;
  if (words > smem_words) {
    bits = scratch + (size_t)(gridDim.x * gridDim.y) * bitmap_words_before(rq.cu, req) + (size_t)(blockIdx.y * gridDim.x + blockIdx.x) * words;
  }
  // the bucket with prefix[d] < b <= prefix[d + 1]
  const int32_t* pf = prefix_all + (((size_t)req * L + layer) * Hkv + g) * (kBins + 1);
  {
    constexpr int PER = kBins / POS_THREADS;
    int at[PER + 1];
#pragma unroll
    for (int q = 0; q < PER; ++q) at[q] = __ldg(&pf[q * POS_THREADS + threadIdx.x]);
    at[PER] = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int next = __ldg(&pf[q * POS_THREADS + threadIdx.x + 1]);
      if (at[q] < b && next >= b) { S.bucket = q * POS_THREADS + threadIdx.x; S.start = at[q]; S.n_in = next - at[q]; }
    }
  }
  if (threadIdx.x == 0) { S.count = 0; S.tie_count = 0; }
  __syncthreads();
  const int d = S.bucket, n_in = S.n_in;
  uint32_t krem = (uint32_t)(b - S.start);           // entries of the bucket that are kept
  uint32_t klo = (uint32_t)(kBins - 1 - d) << (32 - kBinBits), khi = klo | ((1u << (32 - kBinBits)) - 1u);
  const bool listed = n_in <= cap;
  if (listed) {
    // In buckets above zero the bits of a float are compared as they are: as signed integers they have the order of
    // the keys there, and everything else lies below.
    const bool plain = klo > 0x80000000u;
    const int ilo = (int)(klo ^ 0x80000000u), ihi = (int)(khi ^ 0x80000000u);
    const uint4* const v4 = reinterpret_cast<const uint4*>(v - a);
    const int n_oct = (end + 7) >> 3;                // (up to seven elements beyond the row are loaded, and not looked at)
    uint4 next[2];
    auto fetch = [&](int o) {
      next[0] = next[1] = make_uint4(0, 0, 0, 0);
      if (o < n_oct) { next[0] = __ldcg(v4 + 2 * o); next[1] = __ldcg(v4 + 2 * o + 1); }
    };
    fetch(warp * 32 + lane);
    for (int o0 = warp * 32; o0 < n_oct; o0 += POS_THREADS) {
      const int o = o0 + lane;
      uint32_t x[8] = {next[0].x, next[0].y, next[0].z, next[0].w, next[1].x, next[1].y, next[1].z, next[1].w};
      fetch(o + POS_THREADS);
      if (!plain) {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = ordered_key(__uint_as_float(x[e])) ^ 0x80000000u;
      }
      uint32_t above = 0, in = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        above |= (int)x[e] > ihi ? 1u << e : 0u;
        in |= (int)x[e] >= ilo ? 1u << e : 0u;
      }
      // elements of the row among the eight
      const int lo_e = max(0, a - 8 * o), hi_e = min(8, max(0, end - 8 * o));
      const uint32_t row = (0xFFu << lo_e) & (0xFFu >> (8 - hi_e));
      above &= row;
      in &= row & ~above;
      if (o < n_oct) reinterpret_cast<uint8_t*>(bits)[o] = (uint8_t)above;
      if (!__any_sync(0xffffffffu, in != 0)) continue;
      const int mine = __popc(in);
      int inc = mine;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, s);
        if (lane >= s) inc += t;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&S.count, inc);
      at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (in >> e & 1u) list[at++] = make_uint2(x[e] ^ 0x80000000u, (uint32_t)(8 * o + e));
    }
    if (threadIdx.x < 4 && n_oct + (int)threadIdx.x < 4 * words) reinterpret_cast<uint8_t*>(bits)[n_oct + threadIdx.x] = 0;
  }
  __threadfence_block();
  __syncthreads();
  const int cnt = listed ? n_in : n;
  // f(key, element, whether there is such an entry), whole warps
  auto for_entries = [&](auto f) {
    for (int i0 = warp * 32 * SP_BATCH; i0 < cnt; i0 += WARPS * 32 * SP_BATCH) {
      uint2 x[SP_BATCH];
#pragma unroll
      for (int u = 0; u < SP_BATCH; ++u) {
        const int i = i0 + 32 * u + lane;
        x[u] = make_uint2(0u, 0u);
        if (i < cnt) x[u] = listed ? list[i] : make_uint2(ordered_key(__ldcg(v + i)), (uint32_t)(a + i));
      }
#pragma unroll
      for (int u = 0; u < SP_BATCH; ++u)
        if (i0 + 32 * u < cnt) f(x[u].x, (int)x[u].y, i0 + 32 * u + lane < cnt);
    }
  };
  uint32_t n_bin = (uint32_t)n_in;
  while (n_bin > (uint32_t)kFewEntries && klo < khi) {
    const uint32_t width = khi - klo;
    const int shift = width < SP_BINS ? 0 : 22 - __clz(width);
    clear_hist(S);
    for_entries([&](uint32_t key, int, bool have) {
      count_bin(have && key >= klo && key <= khi ? (int)((key - klo) >> shift) : -1, S);
    });
    __syncthreads();
    find_bin(krem, S);
    klo += S.sel_bin << shift;
    if (khi - klo >= 1u << shift) khi = klo + ((1u << shift) - 1u);
    krem = S.sel_rem;
    n_bin = S.sel_cnt;
    __syncthreads();
  }
  // every entry above the bin, and krem of its n_bin entries
  int pos_cut = -1;                                  // more than kTieCap are equal: up to this position
  const bool few = n_bin <= (uint32_t)kTieCap;
  if (!few) {
    int plo = a, phi = end - 1;                      // smallest cut with count(pos <= cut) >= krem
    while (plo < phi) {
      const int mid = plo + ((phi - plo) >> 1);
      int c = 0;
      for_entries([&](uint32_t key, int pos, bool have) { c += have && key == klo && pos <= mid ? 1 : 0; });
      block_excl_scan(c, S.warp_tot, &S.total);
      const int tot = S.total;
      __syncthreads();
      if ((uint32_t)tot >= krem) phi = mid; else plo = mid + 1;
    }
    pos_cut = plo;
  }
  if (!listed) {
    for (int wi = threadIdx.x; wi < words; wi += POS_THREADS) bits[wi] = 0;
    __threadfence_block();
    __syncthreads();
  }
  for_entries([&](uint32_t key, int pos, bool have) {
    if (have && (key > khi || (key == klo && pos <= pos_cut))) atomicOr(&bits[pos >> 5], 1u << (pos & 31));
    if (few && have && key >= klo && key <= khi) S.ties[atomicAdd(&S.tie_count, 1)] = make_uint2(key, (uint32_t)pos);
  });
  __threadfence_block();
  __syncthreads();
  if (few) {
    for (int i = threadIdx.x; i < (int)n_bin; i += POS_THREADS) {
      const uint2 e = S.ties[i];
      uint32_t ahead = 0;
      for (int o = 0; o < (int)n_bin; ++o) {
        const uint2 x = S.ties[o];
        ahead += x.x > e.x || (x.x == e.x && x.y < e.y) ? 1u : 0u;
      }
      if (ahead < krem) atomicOr(&bits[e.y >> 5], 1u << (e.y & 31));
    }
    __threadfence_block();
    __syncthreads();
  }
  int32_t* const dst = row_start();
  for (int t = threadIdx.x; t < Sw; t += POS_THREADS)
    if (b + t < room) dst[b + t] = n + t;
  // Ranks of the bits: a warp takes a run of the words, 32 at a time, so that its lanes write close together.
  const int run = (words + 32 * WARPS - 1) / (32 * WARPS) * 32, w0 = min(words, warp * run), w1 = min(words, w0 + run);
  int ones = 0;
  for (int wi = w0 + lane; wi < w1; wi += 32) ones += __popc(bits[wi]);
  ones = __reduce_add_sync(0xffffffffu, ones);
  if (lane == 0) S.warp_tot[warp] = ones;
  __syncthreads();
  int rank = __reduce_add_sync(0xffffffffu, lane < warp ? S.warp_tot[lane] : 0);
  for (int wb = w0; wb < w1; wb += 32) {
    uint32_t m = wb + lane < w1 ? bits[wb + lane] : 0u;
    const int mine = __popc(m);
    int inc = mine;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, s);
      if (lane >= s) inc += t;
    }
    int at = rank + inc - mine;
    while (m) {
      const int bit = __ffs(m) - 1;
      m &= m - 1;
      if (at < b && at < room) dst[at] = ((wb + lane) << 5) + bit - a;
      ++at;
    }
    rank += __shfl_sync(0xffffffffu, inc, 31);
  }
}

constexpr int GA_THREADS = 128;
constexpr int GA_BATCH = 8;                          // passes of K and of V loads a warp has in flight

// Copies the retained rows, one warp per 32 consecutive packed rows: every lane finds the source of
// one row, then the warp copies them CPR lanes (16 bytes each) to a row.  With dec_off the rows go into
// the decode layout, one spare row (written as zero) behind every head's rows.
//
// Bound: memory; rows of 256 bytes at random places.  One lookup (a binary search and a 64-bit division) per
// row and four rows in flight took 210 us for 1.05 M rows of 256 bytes in K and V (5.1 TB/s).
// Its CTAs take their places while the positions are written out (2 us less per call: four layers of 512 tokens
// 82 -> 80 us); offsets and positions are read behind the wait, so they are not declared read-only here.
template <int CPR, bool kDecode>
__global__ void __launch_bounds__(GA_THREADS)
gather_rows(const LayerPtrs ptrs, const int64_t* offsets, const int64_t* dec_off,
            const int32_t* __restrict__ budget, const int32_t* pos_packed, const ReqInfo* __restrict__ reqs,
            uint4* __restrict__ k_out, uint4* __restrict__ v_out, int n_req, int L, int Hkv, int Sw, int64_t T) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int RPP = 32 / CPR, NIT = 32 / RPP, NB = NIT < GA_BATCH ? NIT : GA_BATCH;
  const int nblk = n_req * L;
  asm volatile("griddepcontrol.wait;" ::: "memory");
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
  const int need_words = (max_n + 3 + 31) / 32;
  const int smem_words = need_words <= kBitmapSmemWords ? (need_words + 1) / 2 * 2 : 0;
  // list of a bucket's entries, 8 bytes each: a sixteenth of the values, or all of a short prompt's
  const int cap = std::min(std::max(2048, max_n / 16), (kSelectSmemWords - smem_words) / 2);
  static PerDeviceOnce attr;
  if (attr.need(ctx->device)) {
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    attr.mark(ctx->device);
  }
  const int64_t ctas = (int64_t)c.n_kv_heads * (hi - lo) * n_req;
  const dim3 grid(c.n_kv_heads, hi - lo, n_req);
  // A list is a chain of scans and short passes: with more lists than the device holds CTAs of 1024
  // threads, smaller ones keep more chains in flight (1024 lists of 4K tokens: 42 us with 1024 threads).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.dynamicSmemBytes = (size_t)(smem_words + 2 * cap) * 4;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = offsets ? 1 : 0;                    // behind run_offsets, which wrote them
  cudaError_t e;
#define CAKE_POSITIONS(NT)                                                                                                \
  cfg.blockDim = dim3(NT);                                                                                                \
  e = cudaLaunchKernelEx(&cfg, sorted_positions<NT>, (const float*)ctx->d_store, (const int32_t*)ctx->d_prefix,           \
                         (const ReqInfo*)ctx->d_req, budget, offsets, out, ctx->d_bitmap, req0, lo,                       \
                         c.n_layers, c.n_kv_heads, c.window, smem_words, cap, ctx->total_tokens, capacity)
  if (ctas <= ctx->n_sm) { CAKE_POSITIONS(1024); }
  else if (ctas <= 2 * ctx->n_sm) { CAKE_POSITIONS(512); }
  else { CAKE_POSITIONS(256); }
#undef CAKE_POSITIONS
  count_launch();
  return cuda_status(e);
}

// Rows of the packed order into k_out / v_out (dec_off: into the decode layout).
int32_t run_gather(cake_ctx* ctx, const LayerPtrs& ptrs, const int64_t* row_off, const int64_t* dec_off, const int32_t* pos,
                   void* k_out, void* v_out, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int32_t* budget = ctx->d_budget[(ctx->n_evicted - 1) & 1];
  const int grid = ctx->n_sm * 5;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(GA_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e;
#define CAKE_GATHER(CPR)                                                                                                 \
  e = cudaLaunchKernelEx(&cfg, dec_off ? gather_rows<CPR, true> : gather_rows<CPR, false>, ptrs, row_off, dec_off, budget, pos,  \
                         (const ReqInfo*)ctx->d_req, (uint4*)k_out, (uint4*)v_out, ctx->n_req, c.n_layers, c.n_kv_heads, \
                         c.window, ctx->total_tokens)
  switch (c.head_dim * (c.dtype == CAKE_DTYPE_FP32 ? 4 : 2) / 16) {
    case 8: CAKE_GATHER(8); break;
    case 16: CAKE_GATHER(16); break;
    default: CAKE_GATHER(32); break;
  }
#undef CAKE_GATHER
  count_launch();
  return cuda_status(e);
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
