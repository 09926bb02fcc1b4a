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

constexpr int kTieCap = 512;                         // entries that can be ranked one by one
constexpr int kFewEntries = 64;                      // entries that are ranked without another histogram
constexpr int SP_BINS = 1024;                        // (22 - clz in the code is 32 - clz - log2 of this)
constexpr int SP_BATCH = 4;                          // groups of 32 entries a warp has in flight
constexpr int SP_UNLISTED = 8;                       // the same of values, where it goes over them again
constexpr int SP_GROUPS = 4;                         // 16-byte groups of values a lane has in flight
constexpr int SP_QUEUE_WORDS = 64 * 5;               // a warp's queue
constexpr int kSelectCluster = kPortableCluster;     // most CTAs that share a list

struct SelectSmem {
  uint32_t hist[2][SP_BINS];                         // in turn: peers read one while the next is counted
  uint2 ties[kTieCap];                               // (key, position)
  int warp_tot[32];
  int total;
  int count, tie_count, ones, before;
  uint32_t sel_bin, sel_rem, sel_cnt;
};
static_assert(sizeof(uint2) * kTieCap <= sizeof(uint32_t) * 2 * SP_BINS, "the cluster's ties take the histograms' place");

// Bins of the histogram, summed over the list's CTAs, from the top: the one that holds the krem-th entry, how many of
// its entries are wanted, and its size.
__device__ inline void find_bin(uint32_t krem, const uint32_t* hist, int csize, SelectSmem& S) {
  constexpr int MOST = SP_BINS / 256;                // bins of a thread
  const int per = max(1, SP_BINS / (int)blockDim.x);
  int h[MOST], mine = 0;
#pragma unroll
  for (int q = 0; q < MOST; ++q) {
    h[q] = 0;
    if (q < per) {
      const uint32_t* at = &hist[SP_BINS - 1 - (threadIdx.x * per + q)];
      if (csize == 1) h[q] = (int)*at;
      else for (int r = 0; r < csize; ++r) h[q] += (int)ld_peer(at, (uint32_t)r);
    }
    mine += h[q];
  }
  int above = block_excl_scan(mine, S.warp_tot, &S.total);
#pragma unroll
  for (int q = 0; q < MOST; ++q) {
    if ((uint32_t)above < krem && (uint32_t)(above + h[q]) >= krem) {
      S.sel_bin = (uint32_t)(SP_BINS - 1 - (threadIdx.x * per + q));
      S.sel_rem = krem - (uint32_t)above;
      S.sel_cnt = (uint32_t)h[q];
    }
    above += h[q];
  }
  __syncthreads();
}
// Counts a bin for every lane that has one (>= 0).  Pooled values repeat: a run of equal bins in
// neighbouring lanes is counted once.  Called by whole warps.
__device__ __forceinline__ void count_bin(int bin, uint32_t* hist) {
  if (!__any_sync(0xffffffffu, bin >= 0)) return;
  const int lane = threadIdx.x & 31, before = __shfl_up_sync(0xffffffffu, bin, 1);
  const bool first = lane == 0 || bin != before;
  const uint32_t firsts = __ballot_sync(0xffffffffu, first);
  if (first && bin >= 0) {
    const uint32_t later = lane < 31 ? firsts >> (lane + 1) : 0u;
    atomicAdd(&hist[bin], later ? (uint32_t)__ffs(later) : 32u - lane);
  }
}

// `csize` CTAs (a cluster) per (head, layer in [lo, hi), request): which positions the current budget b keeps, then
// these in ascending order, then the window, written at out[base + g*len ...].  A CTA owns a run of the values.
//   1. The bucket offsets say which bucket holds the b-th largest value, and how many of its entries are wanted.
//   2. One pass over the values' codes (upper halves of their keys): the bits of those in the buckets before are set, those
//      inside go to the CTA's list in shared memory, as (value, position).  A CTA whose list overflows goes over its
//      values again in the steps below.
//   3. Histograms of SP_BINS equal parts of the bucket's keys, and of the positions where the keys are equal, narrow it to
//      the bin that holds the b-th entry, until that has few entries (usually at once); these are ranked by (key, position).
//   4. Ranks of the bits, positions.
// Bound: the pass over the codes, and between the steps the latency of the chain, which other lists' CTAs on the SM
// hide.  A retained set may be read after every stage, and by layers, so what counts is few lists as much as many, and
// values that share a bucket: 8 lists of 131 040 values 16 us, 80 20, 256 33, 256 of 32 736 17, 1024 of 4064 21; 256 lists whose
// values all share a bucket 206, all equal 370.  With one CTA per list, a pass over the values themselves (lanes 32
// bytes apart, every sector fetched twice), eight buckets to a power of two everywhere and a bisection among equal
// values these took 23, 25, 42, 19, 21, 447 and 2620 us, and ordinary indicators (log-normal, sigma 0.15) overflowed the
// list: 50 us instead of 36 at 256 lists.  Without the bucket offsets three digit histograms of all values took 300 us.
// `bits` is shared memory when a CTA's bits fit, else a slice of global scratch.
template <int POS_THREADS>
__global__ void __launch_bounds__(POS_THREADS, 1024 / POS_THREADS)
sorted_positions(const float* __restrict__ store, const uint16_t* __restrict__ codes, const int32_t* __restrict__ prefix_all, const ReqInfo* __restrict__ reqs, const int32_t* __restrict__ budget,
                 const int64_t* __restrict__ offsets, int32_t* __restrict__ out, uint32_t* __restrict__ scratch,
                 int req0, int lo, int L, int Hkv, int Sw, int csize, int smem_words, int cap, int64_t T,
                 int64_t code_T, int64_t capacity) {
  extern __shared__ __align__(16) uint32_t sh_dyn[];
  __shared__ SelectSmem S;
  const int g = blockIdx.x / csize, rank = blockIdx.x - g * csize, layer = lo + blockIdx.y, req = req0 + blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int WARPS = POS_THREADS / 32;
  const bool split = csize > 1;
  auto meet = [&]() { if (split) cluster_sync(); else __syncthreads(); };
  const ReqInfo rq = reqs[req];
  const int n = rq.n;
  const int b = budget[(size_t)req * L + layer];
  const int len = b + Sw;
  constexpr int PER = kBins / 32, EACH = PER / 32;
  const int32_t* pf = prefix_all + (((size_t)req * L + layer) * Hkv + g) * (kBins + 1);
  const int coarse = __ldg(&pf[PER * lane]);         // (for step 1, on its way with the budget)
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
    const int t0 = rank * POS_THREADS + threadIdx.x, step = csize * POS_THREADS;
    for (int t = t0; t < (b <= 0 ? 0 : n); t += step)
      if (t < room) dst[t] = t;
    for (int t = t0; t < Sw; t += step)
      if (b + t < room) dst[b + t] = n + t;
    return;
  }
  const float* const v = store + ((size_t)layer * Hkv + g) * T + rq.cu;
  // this CTA's words of 32 values, [w_lo, w_hi)
  const int words = (n + 31) >> 5, share = (words + csize - 1) / csize;
  const int w_lo = min(words, rank * share), w_hi = min(words, w_lo + share);
  uint4* const queue = reinterpret_cast<uint4*>(sh_dyn) + warp * 64;             // octets of the warp that are to be taken,
  int* const queue_at = reinterpret_cast<int*>(sh_dyn) + WARPS * 256 + warp * 64;   //   up to 63, and their numbers
  uint32_t* bits = sh_dyn + SP_QUEUE_WORDS * WARPS;
  uint2* const list = reinterpret_cast<uint2*>(bits + smem_words);
  if (share > smem_words)
    bits = scratch + (size_t)(Hkv * gridDim.y) * bitmap_words_before(rq.cu, req) + (size_t)(blockIdx.y * Hkv + g) * words + w_lo;
  // octets (groups of eight values) of this CTA; the last one's codes beyond the prompt are not looked at
  const int o_lo = 4 * w_lo, o_hi = max(o_lo, min((n + 7) >> 3, 4 * w_hi));
  const int o_first = o_lo + warp * 32 * SP_GROUPS + lane;
  const uint4* const c8 = reinterpret_cast<const uint4*>(codes + ((size_t)layer * Hkv + g) * code_T + code_row(rq.cu, req));
  uint4 next[SP_GROUPS];                             // octets of the lane on their way
  auto fetch = [&](int o0) {
#pragma unroll
    for (int u = 0; u < SP_GROUPS; ++u) next[u] = o0 + 32 * u < o_hi ? __ldcg(c8 + o0 + 32 * u) : make_uint4(0, 0, 0, 0);
  };
  fetch(o_first);
  if (threadIdx.x == 0) S.count = S.tie_count = S.ones = S.before = 0;
  for (int wi = threadIdx.x; wi < w_hi - w_lo; wi += POS_THREADS) bits[wi] = 0;
  // The bucket with prefix[d] < b <= prefix[d + 1], by every warp for itself: the 128 that hold it, then the one.
  int bucket, start, n_in;
  {
    const int from = 31 - __clz((int)__ballot_sync(0xffffffffu, coarse < b));          // (prefix[0] = 0 < b)
    int at[EACH], below = 0;
#pragma unroll
    for (int q = 0; q < EACH; ++q) at[q] = __ldg(&pf[PER * from + 32 * q + lane + 1]);
#pragma unroll
    for (int q = 0; q < EACH; ++q) below += __popc(__ballot_sync(0xffffffffu, at[q] < b));
    start = __shfl_sync(0xffffffffu, coarse, from);
    int next = 0;
#pragma unroll
    for (int q = 0; q < EACH; ++q) {
      const int before = __shfl_sync(0xffffffffu, at[q], (below - 1) & 31), after = __shfl_sync(0xffffffffu, at[q], below & 31);
      if (below > 0 && (below - 1) >> 5 == q) start = before;
      if (below >> 5 == q) next = after;
    }
    bucket = PER * from + below;
    n_in = next - start;
  }
  uint32_t krem = (uint32_t)(b - start);             // entries of the bucket that are kept
  uint32_t klo = bucket_first_key(bucket), khi = bucket_last_key(bucket);
  const uint32_t in_lo = klo, in_hi = khi;
  __threadfence_block();
  __syncthreads();
  {
    // One pass over the upper halves of the keys: those above the bucket's are kept, those of the bucket are listed.  Few
    // octets have either; they are gathered in the warp's queue and taken 32 at a time.
    const uint32_t c_lo = klo >> 16, c_hi = khi >> 16;
    auto take = [&](int i, bool have) {
      const int o = queue_at[i & 63];
      const uint4 c = queue[i & 63];
      const uint32_t x[4] = {c.x, c.y, c.z, c.w};
      uint32_t above = 0, in = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t code = e & 1 ? x[e >> 1] >> 16 : x[e >> 1] & 0xFFFFu;
        above |= code > c_hi ? 1u << e : 0u;
        in |= code >= c_lo ? 1u << e : 0u;
      }
      const uint32_t row = have ? 0xFFu >> (8 - min(8, n - 8 * o)) : 0u;         // those of the prompt
      above &= row;
      in &= row & ~above;
      if (above) reinterpret_cast<uint8_t*>(bits)[o - o_lo] = (uint8_t)above;
      const int mine = __popc(in);
      if (!__any_sync(0xffffffffu, mine)) return;
      int inc = mine;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, s);
        if (lane >= s) inc += t;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&S.count, inc);
      at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
      while (in) {
        const int e = __ffs(in) - 1;
        in &= in - 1;
        if (at < cap) {
          list[at].y = (uint32_t)(8 * o + e);
          copy_async4(&list[at].x, v + 8 * o + e);
        }
        ++at;
      }
    };
    int head = 0, tail = 0;
    constexpr int step = POS_THREADS * SP_GROUPS;
    for (int o0 = o_first; o0 - lane < o_hi; o0 += step) {
      uint4 now[SP_GROUPS];
#pragma unroll
      for (int u = 0; u < SP_GROUPS; ++u) now[u] = next[u];
      fetch(o0 + step);
#pragma unroll
      for (int u = 0; u < SP_GROUPS; ++u) {
        const uint32_t most = __vmaxu2(__vmaxu2(now[u].x, now[u].y), __vmaxu2(now[u].z, now[u].w));
        const bool hit = max(most & 0xFFFFu, most >> 16) >= c_lo && o0 + 32 * u < o_hi;
        const uint32_t hits = __ballot_sync(0xffffffffu, hit);
        if (hit) {
          const int i = (tail + __popc(hits & ((1u << lane) - 1u))) & 63;
          queue[i] = now[u];
          queue_at[i] = o0 + 32 * u;
        }
        tail += __popc(hits);
        if (tail - head >= 32) {
          __syncwarp();
          take(head + lane, true);
          head += 32;
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (tail > head) take(head + lane, lane < tail - head);
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __threadfence_block();
  __syncthreads();
  const int cnt = S.count;
  const bool listed = cnt <= cap;
  // f(key, position, whether there is such an entry) for the bucket's entries among this CTA's values, whole warps
  auto for_entries = [&](auto f) {
    if (listed) {
      for (int i0 = warp * 32 * SP_BATCH; i0 < cnt; i0 += WARPS * 32 * SP_BATCH) {
        uint2 x[SP_BATCH];
#pragma unroll
        for (int u = 0; u < SP_BATCH; ++u) x[u] = i0 + 32 * u + lane < cnt ? list[i0 + 32 * u + lane] : make_uint2(0u, 0u);
#pragma unroll
        for (int u = 0; u < SP_BATCH; ++u)
          if (i0 + 32 * u < cnt) f(ordered_key(__uint_as_float(x[u].x)), (int)x[u].y, i0 + 32 * u + lane < cnt);
      }
    } else {
      const int hi_v = min(n, 32 * w_hi);
      for (int i0 = 32 * w_lo + warp * 32 * SP_UNLISTED; i0 < hi_v; i0 += POS_THREADS * SP_UNLISTED) {
        float x[SP_UNLISTED];
#pragma unroll
        for (int u = 0; u < SP_UNLISTED; ++u) x[u] = i0 + 32 * u + lane < hi_v ? __ldcg(v + i0 + 32 * u + lane) : 0.f;
#pragma unroll
        for (int u = 0; u < SP_UNLISTED; ++u) {
          const uint32_t key = ordered_key(x[u]);
          f(key, i0 + 32 * u + lane, i0 + 32 * u + lane < hi_v && key >= in_lo && key <= in_hi);
        }
      }
    }
  };
  // The entries in question: n_bin of them with keys klo to khi and, where these are equal, positions plo to phi.  Those
  // before (larger keys, or equal keys and lower positions) are kept, and krem of the n_bin.
  uint32_t n_bin = (uint32_t)n_in;
  int plo = 0, phi = n - 1;
  const uint32_t few = n_in <= cap ? kFewEntries : kTieCap;      // (a round is a pass over the values if a list has overflowed)
  for (int round = 0; n_bin > few && (krem < n_bin || klo == 0); ++round) {
    uint32_t* const hist = S.hist[round & 1];
    for (int i = threadIdx.x; i < SP_BINS; i += POS_THREADS) hist[i] = 0;
    __syncthreads();
    const bool by_key = klo < khi;
    const uint32_t width = by_key ? khi - klo : (uint32_t)(phi - plo);
    const int shift = width < SP_BINS ? 0 : 22 - __clz(width);
    for_entries([&](uint32_t key, int pos, bool have) {
      const bool in = have && key >= klo && key <= khi && pos >= plo && pos <= phi;
      count_bin(in ? (int)((by_key ? key - klo : (uint32_t)(phi - pos)) >> shift) : -1, hist);
    });
    meet();
    find_bin(krem, hist, csize, S);
    krem = S.sel_rem;
    n_bin = S.sel_cnt;
    const uint32_t at = S.sel_bin << shift, last = (1u << shift) - 1u;
    if (by_key) {
      klo += at;
      khi = min(khi, klo + min(last, 0xFFFFFFFFu - klo));
    } else {
      phi -= (int)at;
      plo = max(plo, phi - (int)last);
    }
  }
  if (krem == n_bin && klo > 0) {                    // all of them are kept
    if (klo < khi) khi = klo - 1u;
    else plo = phi + 1;
    n_bin = 0;
  }
  for_entries([&](uint32_t key, int pos, bool have) {
    const bool kept = key > khi || (key == khi && pos < plo);
    if (have && kept) atomicOr(&bits[(pos >> 5) - w_lo], 1u << (pos & 31));
    if (have && !kept && key >= klo && pos <= phi) S.ties[atomicAdd(&S.tie_count, 1)] = make_uint2(key, (uint32_t)pos);
  });
  __threadfence_block();
  __syncthreads();
  // the cluster's ties, and the kept positions before this CTA's
  uint2* all = S.ties;
  int before = 0;
  if (split) {
    int ones = 0;
    for (int wi = threadIdx.x; wi < w_hi - w_lo; wi += POS_THREADS) ones += __popc(bits[wi]);
    ones = __reduce_add_sync(0xffffffffu, ones);
    if (lane == 0 && ones) atomicAdd(&S.ones, ones);
    meet();
    all = reinterpret_cast<uint2*>(&S.hist[0][0]);
    int at = 0;
    for (int r = 0; r < csize; ++r) {
      const int c = (int)ld_peer(&S.tie_count, (uint32_t)r);
      if (r < rank) before += (int)ld_peer(&S.ones, (uint32_t)r);
      for (int i = threadIdx.x; i < c; i += POS_THREADS) all[at + i] = ld_peer2(&S.ties[i], (uint32_t)r);
      at += c;
    }
    cluster_arrive();                                // nothing of the peers is read from here on
    __syncthreads();
  }
  for (int i = threadIdx.x; i < (int)n_bin; i += POS_THREADS) {
    const uint2 e = all[i];
    uint32_t ahead = 0;
    for (int o = 0; o < (int)n_bin; ++o) {
      const uint2 x = all[o];
      ahead += x.x > e.x || (x.x == e.x && x.y < e.y) ? 1u : 0u;
    }
    const int wi = (int)(e.y >> 5);
    if (ahead < krem && wi >= w_lo && wi < w_hi) atomicOr(&bits[wi - w_lo], 1u << (e.y & 31));
    if (ahead < krem && wi < w_lo) atomicAdd(&S.before, 1);
  }
  __threadfence_block();
  __syncthreads();
  before += S.before;
  int32_t* const dst = row_start();
  if (rank == 0)
    for (int t = threadIdx.x; t < Sw; t += POS_THREADS)
      if (b + t < room) dst[b + t] = n + t;
  // Ranks of the bits: a thread takes a run of the words, or of their bytes where there are more threads than words.
  const int limit = (int)min((int64_t)b, max(room, (int64_t)0));
  auto place = [&](int width, auto unit) {
    const int units = (w_hi - w_lo) * (32 / width), run = (units + POS_THREADS - 1) / POS_THREADS;
    const int u0 = min(units, (int)threadIdx.x * run), u1 = min(units, u0 + run);
    int ones = 0;
    for (int u = u0; u < u1; ++u) ones += __popc(unit(u));
    int to = before + block_excl_scan(ones, S.warp_tot, &S.total);
    for (int u = u0; u < u1; ++u)
      for (uint32_t m = unit(u); m; m &= m - 1, ++to)
        if (to < limit) dst[to] = 32 * w_lo + width * u + __ffs(m) - 1;
  };
  if (w_hi - w_lo < POS_THREADS) place(8, [&](int u) { return (uint32_t)reinterpret_cast<const uint8_t*>(bits)[u]; });
  else place(32, [&](int u) { return bits[u]; });
  if (split) cluster_wait();                         // a peer may still read this CTA's ties
}

constexpr int GA_THREADS = 128;
constexpr int GA_BATCH = 8;                          // passes of K and of V loads a warp has in flight

// Copies the retained rows, one warp per 32 consecutive packed rows: every lane finds the source of
// one row, then the warp copies them CPR lanes (16 bytes each) to a row.  With dec_off the rows go into
// the decode layout, one spare row (written as zero) behind every head's rows.
//
// Bound: memory; rows of 256 bytes at random places.  One lookup (a binary search and a 64-bit division) per
// row and four rows in flight took 210 us for 1.05 M rows of 256 bytes in K and V (5.1 TB/s).
// A short gather's CTAs take their places while the positions are written out (see run_gather); offsets and positions are
// read behind the wait, so they are not declared read-only here.
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
  static PerDeviceOnce attr;
  if (attr.need(ctx->device)) {
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(sorted_positions<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectSmemWords * 4));
    attr.mark(ctx->device);
  }
  const int64_t lists = (int64_t)c.n_kv_heads * (hi - lo) * n_req;
  // Threads per list: as many as the device holds at 1024 per SM, and no more than leave a lane two octets: first in larger
  // CTAs (256 lists of 131 040 values: 33 us with 512 threads, 39 with 256, 41 with 1024), then in more of them (8 lists:
  // 21 us with one CTA of 1024, 16 with eight).
  const int64_t most = std::max<int64_t>((int64_t)ctx->n_sm * 1024 / lists, 256), want = (max_n + 15) / 16;
  int threads = 256, csize = 1;
  while (threads < 1024 && 2 * threads <= most && threads < want) threads *= 2;
  const int widest = widest_cluster(false, kSelectCluster);
  while (2 * csize <= widest && (int64_t)2 * csize * threads <= most && csize * threads < want) csize *= 2;
  // a CTA's bitmap, and its list of the bucket's entries, 8 bytes each: a sixteenth of the values, or all of a short prompt's
  const int share = ((max_n + 31) / 32 + csize - 1) / csize, queue_words = SP_QUEUE_WORDS * threads / 32;
  const int smem_words = share <= kBitmapSmemWords ? (share + 1) / 2 * 2 : 0;
  const int cap = std::min(std::max(2048, 2 * share), (kSelectSmemWords - queue_words - smem_words) / 2);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(c.n_kv_heads * csize), hi - lo, n_req);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)(queue_words + smem_words + 2 * cap) * 4;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  cfg.numAttrs = 0;
  if (offsets) {                                     // behind run_offsets, which wrote them
    at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (csize > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = (unsigned)csize;
    at[cfg.numAttrs].val.clusterDim.y = 1;
    at[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  const cudaError_t e = cudaLaunchKernelEx(&cfg, threads == 1024 ? sorted_positions<1024> : threads == 512 ? sorted_positions<512> : sorted_positions<256>,
                                           (const float*)ctx->d_store, (const uint16_t*)ctx->d_codes, (const int32_t*)ctx->d_prefix, (const ReqInfo*)ctx->d_req, budget, offsets,
                                           out, ctx->d_bitmap, req0, lo, c.n_layers, c.n_kv_heads, c.window, csize, smem_words, cap,
                                           ctx->total_tokens, code_tokens(ctx->total_tokens, ctx->n_req), capacity);
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
  // An early start spares 2 us (four layers of 512 tokens 81.4 -> 78.6 us), but the CTAs then lie where the kernel before had
  // left room and not evenly, which a long gather pays for: 1.05 M rows behind 256 lists of 131 040 values 187 -> 200 us for
  // both, the 128K prefill 4110 -> 4145, a ragged batch 9346 -> 9384; between 131 K and 1 M rows of shorter prompts it is
  // even.  So it is for gathers of up to four runs of 32 rows a warp.
  cfg.numAttrs = ctx->packed_rows_bound <= (int64_t)grid * GA_THREADS ? 1 : 0;
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
