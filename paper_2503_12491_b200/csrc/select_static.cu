// A stand-alone per-head top-k selection that allocates nothing: the entry point for
// callers that must not touch the device allocator.  All its working memory is the shared memory of
// the CTAs that do the work.
#include "cake_internal.cuh"

#include <algorithm>

namespace cake {
namespace {

constexpr int SEL_THREADS = 512;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int kSelMaxWords = 32768;            // limit of the entry point: heads * ceil(n/32)
constexpr int SEL_BINS = 2048;                 // digits of 11, 11 and 10 bits
constexpr int SEL_CLUSTER = kPortableCluster;  // most CTAs per head; SEL_CLUSTER_WIDE where few heads leave SMs idle
constexpr int SEL_CLUSTER_WIDE = 16;           //   and the device holds such a cluster
constexpr int SEL_WIDE_CTAS = 128;             // CTAs (one per SM) up to which clusters of SEL_CLUSTER_WIDE are taken
constexpr int kSelShare = 2048;                // values per CTA below which a head is spread no further
constexpr int kSelSmemKeys = 40 * 1024;        // keys a CTA holds in shared memory; a larger share is read again

__device__ __forceinline__ void st_peer2(const void* p, uint32_t rank, uint2 v) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(peer_addr(p, rank)), "r"(v.x), "r"(v.y) : "memory");
}

// A cluster of `csize` CTAs per head keeps the `keep` entries that come first in the order (value
// descending, position ascending) -- the TopK of Eq. 12 -- and writes their positions in ascending
// order.  Every CTA owns a run of the head's values and holds their keys in shared memory, so the
// values are read once.  Three digit histograms find the key of the keep-th largest entry.  A
// histogram is summed over the cluster by sections: a CTA fetches its section of the bins from every
// CTA's shared memory, adds them up and stores the sums into every CTA's (fetching all bins of all
// CTAs moves csize times as much and took 6 us per histogram at 16 CTAs).  A warp then counts and places
// a run of its own.
//
// Bound: latency (three rounds of histogram, cluster barrier and scan).  One CTA per head that read the
// values from L2 six times and walked its histograms with one thread took 101 us for 8 heads of
// 131 040 values.
__global__ void __launch_bounds__(SEL_THREADS)
select_positions_static(const float* __restrict__ values, int n, int keep, int32_t* __restrict__ out, int csize, int share) {
  extern __shared__ uint32_t keys[];
  __shared__ __align__(16) uint32_t hist[3][SEL_BINS], sums[SEL_BINS];
  __shared__ __align__(16) uint2 parts[SEL_BINS / 2];
  __shared__ uint32_t s_warp[SEL_WARPS];
  __shared__ uint2 s_warp2[SEL_WARPS];
  __shared__ uint32_t s_digit, s_rem;
  __shared__ uint2 x_count[SEL_CLUSTER_WIDE];        // (above, equal) of every CTA of the cluster
  const int rank = (int)cluster_rank();
  const int head = blockIdx.x / csize;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lo = min(n, rank * share), cnt = min(n, lo + share) - lo;
  const float* v = values + (size_t)head * n + lo;
  const bool held = cnt <= kSelSmemKeys;
  for (int i = threadIdx.x; i < 3 * SEL_BINS; i += SEL_THREADS) (&hist[0][0])[i] = 0;
  __syncthreads();
  uint32_t prefix = 0, mask = 0, krem = (uint32_t)keep;
#pragma unroll 1
  for (int round = 0; round < 3; ++round) {
    const int shift = round == 0 ? 21 : round == 1 ? 10 : 0;
    uint32_t* h = hist[round];
    for (int i0 = 0; i0 < cnt; i0 += SEL_THREADS * 8) {
      uint32_t k[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * SEL_THREADS + (int)threadIdx.x;
        k[u] = i < cnt ? (round > 0 && held ? keys[i] : ordered_key(__ldg(&v[i]))) : 0u;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * SEL_THREADS + (int)threadIdx.x;
        if (round == 0 && held && i < cnt) keys[i] = k[u];
        // pooled values repeat: a run of equal digits in neighbouring lanes is counted once
        const uint32_t digit = i < cnt && (k[u] & mask) == prefix ? (k[u] >> shift) & (SEL_BINS - 1) : SEL_BINS;
        if (!__any_sync(0xffffffffu, digit < SEL_BINS)) continue;
        const uint32_t before = __shfl_up_sync(0xffffffffu, digit, 1);
        const bool first = lane == 0 || digit != before;
        const uint32_t firsts = __ballot_sync(0xffffffffu, first);
        if (first && digit < SEL_BINS) {
          const uint32_t later = lane < 31 ? firsts >> (lane + 1) : 0u;
          atomicAdd(&h[digit], later ? (uint32_t)__ffs(later) : 32u - lane);
        }
      }
    }
    const uint32_t* sum = h;
    if (csize > 1) {
      sum = sums;
      cluster_sync();
      const int pairs = SEL_BINS / 2 / csize;        // pairs of bins in a section
      for (int i = threadIdx.x; i < SEL_BINS / 2; i += SEL_THREADS)
        parts[i] = ld_peer2(&h[2 * (rank * pairs + i % pairs)], (uint32_t)(i / pairs));
      __syncthreads();
      if ((int)threadIdx.x < pairs) {
        uint2 t = make_uint2(0, 0);
        for (int p = 0; p < csize; ++p) { t.x += parts[p * pairs + threadIdx.x].x; t.y += parts[p * pairs + threadIdx.x].y; }
        parts[threadIdx.x] = t;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < SEL_BINS / 2; i += SEL_THREADS)
        st_peer2(&sums[2 * (rank * pairs + i % pairs)], (uint32_t)(i / pairs), parts[i % pairs]);
      cluster_sync();
    } else {
      __syncthreads();
    }
    // digits from the top: thread t owns 2047 - 4t .. 2044 - 4t
    constexpr int kOwn = SEL_BINS / SEL_THREADS;
    static_assert(kOwn == 4, "one vector load per thread");
    const int d0 = SEL_BINS - kOwn - kOwn * (int)threadIdx.x;
    const uint4 c = *reinterpret_cast<const uint4*>(&sum[d0]);
    const uint32_t own = c.x + c.y + c.z + c.w;
    uint32_t inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    uint32_t w = lane < SEL_WARPS ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    const uint32_t base = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
    uint32_t above = (warp ? base : 0u) + inc - own;                 // entries with a larger digit than this thread's
    const uint32_t bins[4] = {c.w, c.z, c.y, c.x};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (above < krem && above + bins[q] >= krem) { s_digit = (uint32_t)(d0 + 3 - q); s_rem = krem - above; }
      above += bins[q];
    }
    __syncthreads();
    prefix |= s_digit << shift;
    krem = s_rem;
    mask |= (uint32_t)(SEL_BINS - 1) << shift;
  }
  const uint32_t thr = prefix;        // key of the keep-th largest entry
  const uint32_t need_eq = krem;      // entries equal to it that are kept: the lowest positions
  // every warp owns a run of the CTA's values: count, then place
  const int per = (cnt + SEL_THREADS - 1) / SEL_THREADS * 32;        // values per warp, whole ballots
  const int w_lo = min(cnt, warp * per), w_hi = min(cnt, w_lo + per);
  uint2 mine = make_uint2(0, 0);
  auto key_at = [&](int i) { return i < w_hi ? (held ? keys[i] : ordered_key(__ldg(&v[i]))) : 0u; };
  for (int i0 = w_lo; i0 < w_hi; i0 += 128) {
    uint32_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = key_at(i0 + 32 * u + lane);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool in = i0 + 32 * u + lane < w_hi;
      mine.x += in && k[u] > thr ? 1u : 0u;
      mine.y += in && k[u] == thr ? 1u : 0u;
    }
  }
  mine.x = __reduce_add_sync(0xffffffffu, mine.x);
  mine.y = __reduce_add_sync(0xffffffffu, mine.y);
  if (lane == 0) s_warp2[warp] = mine;
  __syncthreads();
  uint2 before, total = lane < SEL_WARPS ? s_warp2[lane] : make_uint2(0, 0);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, total.x, o), y = __shfl_up_sync(0xffffffffu, total.y, o);
    if (lane >= o) { total.x += x; total.y += y; }
  }
  before = make_uint2(__shfl_sync(0xffffffffu, total.x, warp) - mine.x, __shfl_sync(0xffffffffu, total.y, warp) - mine.y);
  total = make_uint2(__shfl_sync(0xffffffffu, total.x, 31), __shfl_sync(0xffffffffu, total.y, 31));
  if (csize > 1) {
    if ((int)threadIdx.x < csize) st_peer2(&x_count[rank], threadIdx.x, total);
    cluster_sync();               // also: nobody leaves while its histograms may still be read
    for (int p = 0; p < rank; ++p) { before.x += x_count[p].x; before.y += x_count[p].y; }
  }
  int32_t* dst = out + (size_t)head * keep;
  const uint32_t lt = (1u << lane) - 1u;
  for (int i0 = w_lo; i0 < w_hi; i0 += 128) {
    uint32_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = key_at(i0 + 32 * u + lane);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + 32 * u + lane;
      const uint32_t gt = __ballot_sync(0xffffffffu, i < w_hi && k[u] > thr);
      const uint32_t eq = __ballot_sync(0xffffffffu, i < w_hi && k[u] == thr);
      if (gt | eq) {
        const uint32_t g = before.x + __popc(gt & lt), e = before.y + __popc(eq & lt);
        if ((gt >> lane) & 1u) dst[g + min(e, need_eq)] = lo + i;
        else if (((eq >> lane) & 1u) && e < need_eq) dst[g + e] = lo + i;
        before.x += __popc(gt);
        before.y += __popc(eq);
      }
    }
  }
}

}  // namespace
}  // namespace cake

extern "C" int32_t cake_select_positions_static(const float* values, int32_t n_heads, int32_t n,
                                                int32_t keep, int32_t* positions_out, void* stream) {
  using namespace cake;
  if (n_heads < 0 || n < 0 || keep < 0 || keep > n) return CAKE_ERR_ARG;
  if (n_heads == 0 || keep == 0) return CAKE_OK;
  if (!values || !positions_out) return CAKE_ERR_ARG;
  const int words = (n + 31) / 32;
  if ((int64_t)n_heads * words > kSelMaxWords) return CAKE_ERR_CAPACITY;
  int dev = -1;
  CAKE_CUDA_TRY(cudaGetDevice(&dev));
  static PerDeviceOnce attr;
  static bool fits[kOnceDevices];
  bool wide = dev >= 0 && dev < kOnceDevices && fits[dev];
  if (attr.need(dev)) {
    CAKE_CUDA_TRY(cudaFuncSetAttribute(select_positions_static, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelSmemKeys * 4));
    wide = cluster_fits(select_positions_static, SEL_CLUSTER_WIDE, SEL_THREADS, (size_t)kSelSmemKeys * 4);
    if (dev >= 0 && dev < kOnceDevices) fits[dev] = wide;
    attr.mark(dev);
  }
  // as many CTAs per head as leave each kSelShare values, up to 8, or 16 where that still fits the
  // device side by side (one 512-thread CTA per SM)
  const int widest = widest_cluster(wide, SEL_CLUSTER_WIDE);
  int csize = 1;
  while ((int64_t)csize * kSelShare < n && csize * 2 <= widest &&
         (csize < SEL_CLUSTER || (csize < SEL_CLUSTER_WIDE && n_heads * csize * 2 <= SEL_WIDE_CTAS))) csize *= 2;
  const int share = ((n + csize - 1) / csize + 31) / 32 * 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_heads * csize), 1, 1);
  cfg.blockDim = dim3(SEL_THREADS, 1, 1);
  cfg.dynamicSmemBytes = (size_t)std::min(share, kSelSmemKeys) * 4;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, select_positions_static, values, n, keep, positions_out, csize, share);
  count_launch();
  return cuda_status(e);
}
