// Decode-time eviction with frozen per-layer budgets (Section 5.1 "Implementation Details";
// Appendix "More Implementation Details"; the decode branches of the appendix listing).
//
// After the prefill cascade every (request, layer) keeps len = b + S_w tokens per KV head.  The
// decode cache of a block (request, layer) is laid out [H_kv][cap][d] with cap = len + 1: a head
// owns cap row slots, len of them hold the retained tokens and one is free.  Per generated token
// and layer, cake_decode_step
//   1. writes the new token's K/V row into the head's free slot,
//   2. takes the new query's attention over the head's cap cached keys (softmax over all of
//      them, the columns of the S_w most recent tokens dropped, mean over the group's query heads),
//   3. pools it along ascending token position and updates the stored scores with it,
//   4. evicts the entry that comes last in the order (score descending, position ascending)
//      among the tokens outside the recent window: its slot becomes the free one.
// Rows never move: the order of a head's entries by position is kept as a list of slots.
#include "cake_internal.cuh"

#include <algorithm>
#include <cstdlib>

#include <math_constants.h>

namespace cake {
namespace {

constexpr int DEC_THREADS = 512;
constexpr int DEC_CLUSTER = kPortableCluster;   // most CTAs that share a head in the cluster form of the step kernel,
constexpr int DEC_CLUSTER_WIDE = 16;   //   and the most where the grid is small and the device holds such a cluster
constexpr int DEC_CTA_ENTRIES = 256;       // entries per CTA up to which a head is spread no further
constexpr size_t kDecSmemMax = 200 * 1024;
constexpr int DEC_ROWS = 4;       // cache rows a half-warp has in flight in the logit loop

// One CTA per (head, layer, request): positions (ascending, from the packed order), identity
// slot order, and the stored indicator of every survivor (0 for the window).
__global__ void __launch_bounds__(DEC_THREADS)
decode_build(const float* __restrict__ store, const ReqInfo* __restrict__ reqs,
             const int32_t* __restrict__ budget, const int64_t* __restrict__ packed_off,
             const int32_t* __restrict__ pos_packed, const int64_t* __restrict__ dec_off,
             float* __restrict__ score, int32_t* __restrict__ pos, int32_t* __restrict__ order,
             int4* __restrict__ meta, int L, int Hkv, int Sw, int64_t T) {
  const int g = blockIdx.x, layer = blockIdx.y, req = blockIdx.z;
  const ReqInfo rq = reqs[req];
  const int blk = req * L + layer;
  const int b = budget[blk];
  const int len = b + Sw, cap = len + 1;
  const int32_t* src = pos_packed + packed_off[blk] + (int64_t)g * len;
  const float* values = store + ((size_t)layer * Hkv + g) * T + rq.cu;
  const int64_t base = dec_off[blk] + (int64_t)g * cap;
  for (int i = threadIdx.x; i < cap; i += DEC_THREADS) {
    const int p = i < len ? src[i] : -1;
    const float v = i < b ? values[p] : 0.f;
    pos[base + i] = p;
    order[base + i] = i;
    score[base + i] = v == 0.f ? 0.f : v;              // (-0 is stored as +0)
  }
  if (threadIdx.x == 0) meta[(size_t)blk * Hkv + g] = make_int4(len, len, rq.N, b);
}

struct DecodeArgs {
  const void* q_new;       // [n_req][H_q][d]
  const void* k_new;       // [n_req][H_kv][d]
  const void* v_new;
  void* k_cache;           // decode cache rows of d elements
  void* v_cache;
  const int64_t* dec_off;
  float* score;
  int32_t* pos;
  int32_t* order;
  int4* meta;              // (len, free slot, next position, frozen budget)
  int32_t* status;
  float* tmp;              // per (head, request) work area for heads beyond the shared-memory plan
  const ReqInfo* reqs;
  int64_t T;               // tokens of the batch
  int n_req;
  int layer, L, Hq, Hkv, d, Sw, kp, pool_mode, update_mode, smem_cap;
  float scale2;
};

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

// A lane's share of a row (up to 32 bytes held as four 8-byte words) as eight floats; elements
// beyond the share are zero because the words beyond it are.
template <typename T> __device__ __forceinline__ void unpack_row(const uint2 (&w)[4], float (&out)[8]);
template <> __device__ __forceinline__ void unpack_row<float>(const uint2 (&w)[4], float (&out)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) { out[2 * i] = __uint_as_float(w[i].x); out[2 * i + 1] = __uint_as_float(w[i].y); }
}
template <> __device__ __forceinline__ void unpack_row<__nv_bfloat16>(const uint2 (&w)[4], float (&out)[8]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    out[4 * i] = __uint_as_float(w[i].x << 16);     out[4 * i + 1] = __uint_as_float(w[i].x & 0xFFFF0000u);
    out[4 * i + 2] = __uint_as_float(w[i].y << 16); out[4 * i + 3] = __uint_as_float(w[i].y & 0xFFFF0000u);
  }
}

// (value, index) argmin with the tie rule of the eviction: the lowest score goes, among equal
// scores the highest rank (= the highest token position).
__device__ __forceinline__ void worse_of(float& v, int& i, float ov, int oi) {
  if (ov < v || (ov == v && oi > i)) { v = ov; i = oi; }
}

// One CTA per (KV head, request): heads that the cluster form below does not take (see
// launch_decode_step).  Dynamic shared memory: p[G][cap] (logits, then unnormalised
// probabilities by slot) and abar[cap] (group-mean attention by rank).
template <typename T, int G>
__global__ void __launch_bounds__(DEC_THREADS)
decode_step_kernel(const DecodeArgs A) {
  extern __shared__ float sh[];
  __shared__ float red_v[DEC_THREADS / 32];
  __shared__ int red_i[DEC_THREADS / 32];
  __shared__ float s_m[G], s_z[G];
  const int g = blockIdx.x, req = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int blk = req * A.L + A.layer;
  const size_t lid = (size_t)blk * A.Hkv + g;
  const int4 mt = A.meta[lid];
  const int len = mt.x, fre = mt.y, next_pos = mt.z, budget = mt.w;
  const int cap = len + 1;
  const int64_t base = A.dec_off[blk] + (int64_t)g * cap;
  // A head beyond the shared-memory plan works in global memory: its (G + 1) * cap floats lie
  // at the request's token offset of a [H_kv][tokens + requests] area (cap <= N + 1).
  float* p = cap <= A.smem_cap                       // [G][cap]
                 ? sh
                 : A.tmp + (size_t)(G + 1) * ((size_t)g * (size_t)(A.T + A.n_req) + (size_t)A.reqs[req].cu + req);
  float* abar = p + (size_t)G * cap;                 // [cap]
  T* kc = reinterpret_cast<T*>(A.k_cache) + (size_t)base * A.d;
  T* vc = reinterpret_cast<T*>(A.v_cache) + (size_t)base * A.d;
  const T* kn = reinterpret_cast<const T*>(A.k_new) + ((size_t)req * A.Hkv + g) * A.d;
  const T* vn = reinterpret_cast<const T*>(A.v_new) + ((size_t)req * A.Hkv + g) * A.d;
  // 1. the new token takes the free slot and the last rank
  for (int e = threadIdx.x; e < A.d; e += DEC_THREADS) {
    kc[(size_t)fre * A.d + e] = kn[e];
    vc[(size_t)fre * A.d + e] = vn[e];
  }
  if (threadIdx.x == 0) {
    A.order[base + len] = fre;
    A.pos[base + fre] = next_pos;
  }
  // 2. logits of the G query heads against every slot: 16 lanes per row, two rows per warp pass
  const int sub = lane >> 4, l16 = lane & 15;
  const int per = A.d / 16;                          // elements of a row per lane
  float qv[G][8];
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int e = 0; e < 8; ++e)
      qv[h][e] = e < per ? to_f32(reinterpret_cast<const T*>(A.q_new)[((size_t)req * A.Hq + g * G + h) * A.d +
                                                                     l16 * per + e]) : 0.f;
  // a lane's share of a row is 8, 16 or 32 bytes: 8-byte loads, DEC_ROWS rows in flight per half-warp
  const int n8 = per * (int)sizeof(T) / 8;
  constexpr int kStep = (DEC_THREADS / 32) * 2;
  for (int s0 = warp * 2; s0 < cap; s0 += kStep * DEC_ROWS) {
    uint2 raw[DEC_ROWS][4];
#pragma unroll
    for (int u = 0; u < DEC_ROWS; ++u) {
      const int s = s0 + u * kStep + sub;
      const T* row = s == fre ? kn : kc + (size_t)s * A.d;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        raw[u][i] = (s < cap && i < n8) ? reinterpret_cast<const uint2*>(row + l16 * per)[i] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < DEC_ROWS; ++u) {
      const int s = s0 + u * kStep + sub;
      float kv[8];
      unpack_row<T>(raw[u], kv);
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc = fmaf(qv[h][e], kv[e], acc);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (l16 == 0 && s < cap) p[(size_t)h * cap + s] = acc * A.scale2;
      }
    }
  }
  __syncthreads();
  // 3. softmax per head over all cap slots (base 2)
  for (int h = 0; h < G; ++h) {
    float m = -CUDART_INF_F;
#pragma unroll 4
    for (int s = threadIdx.x; s < cap; s += DEC_THREADS) m = fmaxf(m, p[(size_t)h * cap + s]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red_v[warp] = m;
    __syncthreads();
    m = red_v[0];
    for (int w = 1; w < DEC_THREADS / 32; ++w) m = fmaxf(m, red_v[w]);
    __syncthreads();
    float z = 0.f;
#pragma unroll 4
    for (int s = threadIdx.x; s < cap; s += DEC_THREADS) {
      const float e = exp2f(p[(size_t)h * cap + s] - m);
      p[(size_t)h * cap + s] = e;
      z += e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (lane == 0) red_v[warp] = z;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (int w = 0; w < DEC_THREADS / 32; ++w) t += red_v[w];
      s_z[h] = t;
      s_m[h] = m;
    }
    __syncthreads();
  }
  // 4. group-mean observed attention by rank (ascending position), pooling, score update
  const int n_obs = cap - A.Sw;                      // entries outside the recent window
  const int n_old = len - A.Sw;                      // of which these already carry a score
#pragma unroll 4
  for (int r = threadIdx.x; r < n_obs; r += DEC_THREADS) {
    const int s = A.order[base + r];
    float a = 0.f;
#pragma unroll
    for (int h = 0; h < G; ++h) a += p[(size_t)h * cap + s] / s_z[h];
    abar[r] = a * (1.f / (float)G);
  }
  __syncthreads();
  const int rad = A.kp >> 1;
  float worst = CUDART_INF_F;
  int worst_r = -1;
#pragma unroll 2
  for (int r = threadIdx.x; r < n_obs; r += DEC_THREADS) {
    const int lo = max(0, r - rad), hi = min(n_obs, r + rad + 1);
    float v = abar[lo];
    for (int x = lo + 1; x < hi; ++x) v = A.pool_mode == CAKE_POOL_MAX ? fmaxf(v, abar[x]) : v + abar[x];
    if (A.pool_mode != CAKE_POOL_MAX) v /= (float)A.kp;
    const int s = A.order[base + r];
    float sc = v;
    if (r < n_old) {
      const float old = A.score[base + s];
      sc = A.update_mode == CAKE_DECODE_ADD ? old + v : A.update_mode == CAKE_DECODE_MAX ? fmaxf(old, v) : v;
    }
    A.score[base + s] = sc;
    worse_of(worst, worst_r, sc, r);
  }
  // 5. evict back to the frozen budget: the entry that is last in (score desc, position asc)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, worst, o);
    const int oi = __shfl_xor_sync(0xffffffffu, worst_r, o);
    if (oi >= 0 && (worst_r < 0 || ov < worst || (ov == worst && oi > worst_r))) { worst = ov; worst_r = oi; }
  }
  __syncthreads();                                   // red_v is free again
  if (lane == 0) { red_v[warp] = worst; red_i[warp] = worst_r; }
  __syncthreads();
  int ev = -1;
  if (n_obs > budget) {
    float bv = CUDART_INF_F;
    for (int w = 0; w < DEC_THREADS / 32; ++w) {
      if (red_i[w] >= 0 && (ev < 0 || red_v[w] < bv || (red_v[w] == bv && red_i[w] > ev))) {
        bv = red_v[w];
        ev = red_i[w];
      }
    }
  }
  if (ev < 0) {                                      // below the budget: the cache would have to grow
    if (threadIdx.x == 0) atomicCAS(A.status, 0, CAKE_ERR_CAPACITY);
    return;
  }
  // ranks after the evicted one move down by one; its slot becomes the free one
  const int ev_slot = A.order[base + ev];
  __syncthreads();
  for (int r0 = ev; r0 < cap - 1; r0 += DEC_THREADS * 4) {       // four batches per round trip
    int nxt[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + u * DEC_THREADS + threadIdx.x;
      nxt[u] = r < cap - 1 ? A.order[base + r + 1] : 0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + u * DEC_THREADS + threadIdx.x;
      if (r < cap - 1) A.order[base + r] = nxt[u];
    }
    __syncthreads();                                 // the next round reads beyond what this one wrote, but keep rounds apart
  }
  if (threadIdx.x == 0) {
    A.order[base + cap - 1] = ev_slot;
    A.pos[base + ev_slot] = -1;
    A.meta[lid] = make_int4(len, ev_slot, next_pos + 1, budget);
  }
}

// ---------------------------------------------------------------- the step on a cluster of CTAs
// Stores into the shared memory of CTA `rank` of the cluster, at the place `p` has in this CTA's.
__device__ __forceinline__ void st_remote(const void* p, uint32_t rank, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(peer_addr(p, rank)), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_remote(const void* p, uint32_t rank, uint4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(peer_addr(p, rank)), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

// 32 bytes in one load: with four lanes to a row a load covers whole 128-byte lines, half the L1 tag
// look-ups of 16-byte loads.
__device__ __forceinline__ void ld_32b(const void* p, uint4& a, uint4& b) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(p)
               : "memory");
}

// D[16 rows][8 heads] += A[16][16] B[16][8], bf16 operands, fp32 accumulators.
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Logits (base 2) of the G query heads against the rows of ranks w_lo .. w_lo + n_win - 1 into
// lg[h * stride + i], and every warp's maximum per head.  `ord` holds the ranks' slots; the last rank of the head (`new_i`, if it lies
// in the window) is the new token, whose row comes from k_new.  bf16: a warp takes 16 rows at a
// time, every lane loads whole 16-byte pieces of two rows and uses them as the A operand of
// m16n8k16 MMAs with the contraction index permuted (the query operand has the same permutation),
// so a row costs no conversion, no shuffle and no shared memory.
template <int G>
__device__ __forceinline__ void window_logits(const __nv_bfloat16* kc, const __nv_bfloat16* kn, const __nv_bfloat16* q,
                                              int d, int n_win, const int* ord, int new_i, float scale2, float* lg,
                                              int stride, float (*warp_max)[G]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r8 = lane >> 2, t = lane & 3;
  float m0 = -CUDART_INF_F, m1 = -CUDART_INF_F;
  const int n_c = d / 64;                            // 32-byte pieces of a row per lane: 1 or 2
  uint4 qv[4];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    qv[2 * c] = qv[2 * c + 1] = make_uint4(0, 0, 0, 0);
    if (r8 < G && c < n_c) ld_32b(q + (size_t)r8 * d + (4 * c + t) * 16, qv[2 * c], qv[2 * c + 1]);
  }
  for (int i0 = warp * 16; i0 < n_win; i0 += (DEC_THREADS / 32) * 16) {
    uint4 x[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = i0 + r8 + 8 * u;
      const __nv_bfloat16* row = i == new_i ? kn : kc + (size_t)ord[min(i, n_win - 1)] * d;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        x[u][2 * c] = x[u][2 * c + 1] = make_uint4(0, 0, 0, 0);
        if (c < n_c) ld_32b(row + (4 * c + t) * 16, x[u][2 * c], x[u][2 * c + 1]);
      }
    }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      mma_bf16(acc, x[0][c].x, x[1][c].x, x[0][c].y, x[1][c].y, qv[c].x, qv[c].y);
      mma_bf16(acc, x[0][c].z, x[1][c].z, x[0][c].w, x[1][c].w, qv[c].z, qv[c].w);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = i0 + r8 + 8 * u;
      if (i < n_win) {
        const float l0 = acc[2 * u] * scale2, l1 = acc[2 * u + 1] * scale2;
        m0 = fmaxf(m0, l0);
        m1 = fmaxf(m1, l1);
        if (2 * t < G) lg[(2 * t) * stride + i] = l0;
        if (2 * t + 1 < G) lg[(2 * t + 1) * stride + i] = l1;
      }
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
    m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
  }
  if (r8 == 0) {
    if (2 * t < G) warp_max[warp][2 * t] = m0;
    if (2 * t + 1 < G) warp_max[warp][2 * t + 1] = m1;
  }
}
// fp32: 16 lanes per row, fp32 FMAs.
template <int G>
__device__ __forceinline__ void window_logits(const float* kc, const float* kn, const float* q, int d, int n_win,
                                              const int* ord, int new_i, float scale2, float* lg, int stride,
                                              float (*warp_max)[G]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane >> 4, l16 = lane & 15;
  float m[G];
#pragma unroll
  for (int h = 0; h < G; ++h) m[h] = -CUDART_INF_F;
  const int n4 = d / 64;                             // 16-byte pieces per lane: 1 or 2
  float4 qv[G][2];
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int c = 0; c < 2; ++c)
      qv[h][c] = c < n4 ? reinterpret_cast<const float4*>(q + (size_t)h * d)[16 * c + l16] : make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int kStep = (DEC_THREADS / 32) * 2;
  for (int i0 = warp * 2 + sub; i0 - sub < n_win; i0 += kStep * DEC_ROWS) {
    float4 x[DEC_ROWS][2];
#pragma unroll
    for (int u = 0; u < DEC_ROWS; ++u) {
      const int i = i0 + u * kStep;
      const float* row = i == new_i ? kn : kc + (size_t)ord[min(i, n_win - 1)] * d;
#pragma unroll
      for (int c = 0; c < 2; ++c)
        x[u][c] = c < n4 ? reinterpret_cast<const float4*>(row)[16 * c + l16] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < DEC_ROWS; ++u) {
      const int i = i0 + u * kStep;
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          acc = fmaf(qv[h][c].x, x[u][c].x, acc);
          acc = fmaf(qv[h][c].y, x[u][c].y, acc);
          acc = fmaf(qv[h][c].z, x[u][c].z, acc);
          acc = fmaf(qv[h][c].w, x[u][c].w, acc);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (i < n_win) {
          m[h] = fmaxf(m[h], acc * scale2);
          if (l16 == 0) lg[h * stride + i] = acc * scale2;
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < G; ++h) {
    m[h] = fmaxf(m[h], __shfl_xor_sync(0xffffffffu, m[h], 16));
    if (lane == 0) warp_max[warp][h] = m[h];
  }
}

// (score, rank) as one integer whose minimum is the entry that goes: the lowest score, among equal
// scores the highest rank.  -0 and +0 are equal.
__device__ __forceinline__ unsigned long long evict_key(float score, int rank) {
  uint32_t b = __float_as_uint(score);
  if (b == 0x80000000u) b = 0u;
  b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return ((unsigned long long)b << 32) | (uint32_t)(0x7FFFFFFF - rank);
}
constexpr unsigned long long kNoKey = ~0ull;

// The same step with a head spread over a cluster of `csize` CTAs by RANK: a CTA owns a contiguous
// run of the head's entries in ascending token position and, besides, computes the logits of the
// pool_kernel / 2 neighbours on either side, so pooling needs nothing from the other CTAs.  The
// softmax sums are taken against the CTA's own maximum and corrected once the maxima and sums of
// the cluster are known, so a step meets the cluster twice: (maximum, sum) per
// head, then (score, rank, slot) of the eviction candidate.  The old list of slots stays in shared
// memory from the first read on, so its shift needs no further meeting.
//
// Bound: the latency of one chain per layer and token (state -> slots -> key rows -> two cluster
// barriers -> stores); the keys of a layer (8 MB at budgets of 4096) take 1.3 us at the copy rate, 30 %
// of the issue slots and 10 % of the DRAM rate are used.  A launch by itself takes 11 to 14 us at
// budgets of 4096 and 10 to 11 us for four requests at 768; launches that start early follow one another every
// 8.3 us (128K prompt) to 9.4 us.  Cut by slot with a third meeting for the pooled window, a fourth for
// the list shift, and shuffles for the dot products they followed every 26 us.
// Dynamic shared memory: (G + 3) words per entry of the largest window (logits, mean, slot, score).
template <typename T, int G>
__global__ void __launch_bounds__(DEC_THREADS, 2)
decode_step_cluster_kernel(const DecodeArgs A, int csize, int cap_words) {
  extern __shared__ __align__(16) float sh[];
  __shared__ __align__(16) float2 x_mz[DEC_CLUSTER_WIDE][G];      // (maximum, sum) of every CTA of the cluster
  __shared__ __align__(16) uint4 x_cand[DEC_CLUSTER_WIDE];        // eviction candidate of every CTA: key, slot
  __shared__ float red[DEC_THREADS / 32][G], red_z[DEC_THREADS / 32][G];
  __shared__ float s_m[G];
  __shared__ unsigned long long red_k[DEC_THREADS / 32];
  const int crank = (int)cluster_rank();
  if (csize > 1) cluster_arrive();                   // peers may be written only once they run: waited for below
  const int g = blockIdx.x / csize, req = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int blk = req * A.L + A.layer;
  const size_t lid = (size_t)blk * A.Hkv + g;
  const int4 mt = A.meta[lid];
  const int64_t off = A.dec_off[blk];
  const int len = mt.x, fre = mt.y, next_pos = mt.z, budget = mt.w;
  const int cap = len + 1;
  const int64_t base = off + (int64_t)g * cap;
  const int part = (cap + csize - 1) / csize;
  const int r_lo = min(cap, crank * part), r_hi = min(cap, r_lo + part);
  const int rad = A.kp >> 1;
  const int w_lo = max(0, r_lo - rad), w_hi = r_hi > r_lo ? min(cap, r_hi + max(rad, 1)) : w_lo;
  const int n_win = w_hi - w_lo, own = r_lo - w_lo, n_own = r_hi - r_lo;
  float* lg = sh;                                    // [G][cap_words] logits
  float* abar = lg + (size_t)G * cap_words;          // group-mean attention
  int* ord = reinterpret_cast<int*>(abar + cap_words);
  float* old = reinterpret_cast<float*>(ord + cap_words);
  T* kc = reinterpret_cast<T*>(A.k_cache) + (size_t)base * A.d;
  T* vc = reinterpret_cast<T*>(A.v_cache) + (size_t)base * A.d;
  const T* kn = reinterpret_cast<const T*>(A.k_new) + ((size_t)req * A.Hkv + g) * A.d;
  const T* vn = reinterpret_cast<const T*>(A.v_new) + ((size_t)req * A.Hkv + g) * A.d;
  // 1. slots of the window
  for (int i = threadIdx.x; i < n_win; i += DEC_THREADS) ord[i] = w_lo + i == len ? fre : A.order[base + w_lo + i];
  __syncthreads();
  const int new_i = (w_lo <= len && len < w_hi) ? len - w_lo : -1;
  // the rows on their way to L2 before the first pass over them waits
  for (int i = threadIdx.x; i < n_win; i += DEC_THREADS)
    if (i != new_i)
      for (int b = 0; b < A.d * (int)sizeof(T); b += 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(kc + (size_t)ord[i] * A.d) + b));
  const int n_obs = cap - A.Sw;                      // entries outside the recent window
  const int n_old = len - A.Sw;                      // of which these already carry a score
  for (int i = threadIdx.x; i < n_own; i += DEC_THREADS) old[i] = r_lo + i < n_old ? A.score[base + ord[own + i]] : 0.f;
  // Everything up to here reads the context's own state of this layer; the caller's tensors may
  // come from the kernel before this one in the stream.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // 2. logits of the window's rows
  window_logits<G>(kc, kn, reinterpret_cast<const T*>(A.q_new) + ((size_t)req * A.Hq + g * G) * A.d, A.d, n_win, ord, new_i,
                   A.scale2, lg, cap_words, red);
  __syncthreads();
  // the new token takes the free slot and the last rank
  if (r_lo <= len && len < r_hi) {
    const int n16 = A.d * (int)sizeof(T) / 16;
    if (threadIdx.x < n16)
      reinterpret_cast<uint4*>(kc + (size_t)fre * A.d)[threadIdx.x] = reinterpret_cast<const uint4*>(kn)[threadIdx.x];
    else if (threadIdx.x < 2 * n16)
      reinterpret_cast<uint4*>(vc + (size_t)fre * A.d)[threadIdx.x - n16] = reinterpret_cast<const uint4*>(vn)[threadIdx.x - n16];
    if (threadIdx.x == 0) A.pos[base + fre] = next_pos;
  }
  // 3. maximum of the window and sum of the CTA's own entries, per head (base 2)
  {
    float m[G], z[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
      float t = red[lane % (DEC_THREADS / 32)][h];
#pragma unroll
      for (int o = DEC_THREADS / 64; o > 0; o >>= 1) t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, o));
      m[h] = t;
      z[h] = 0.f;
    }
    for (int i = own + threadIdx.x; i < own + n_own; i += DEC_THREADS)
#pragma unroll
      for (int h = 0; h < G; ++h) z[h] += exp2f(lg[h * cap_words + i] - m[h]);
#pragma unroll
    for (int h = 0; h < G; ++h) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z[h] += __shfl_xor_sync(0xffffffffu, z[h], o);
      if (lane == h) red_z[warp][h] = z[h];
      if (threadIdx.x == h) s_m[h] = m[h];
    }
  }
  __syncthreads();
  if (csize > 1) cluster_wait();                     // every CTA of the cluster runs
  if (threadIdx.x < csize * G) {
    const int h = threadIdx.x % G, peer = threadIdx.x / G;
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < DEC_THREADS / 32; ++w) t += red_z[w][h];
    const float2 v = make_float2(s_m[h], t);
    if (csize > 1) st_remote(&x_mz[crank][h], (uint32_t)peer, v);
    else x_mz[0][h] = v;
  }
  if (csize > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
  // 4. group-mean attention along the window, pooling, score update, eviction candidate
  //    (every CTA takes the probabilities from the same maximum and sum: entries that share the
  //    largest neighbour tie exactly, on whichever side of a CTA boundary they lie)
  float gm[G], fac[G];
  {
    // a lane takes head lane % G of every (32 / G)-th CTA
    const int h = lane % G;
    float m = -CUDART_INF_F, z = 0.f;
    for (int c = lane / G; c < csize; c += 32 / G) m = fmaxf(m, x_mz[c][h].x);
#pragma unroll
    for (int o = G; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    for (int c = lane / G; c < csize; c += 32 / G) {
      const float2 v = x_mz[c][h];
      if (v.y > 0.f) z += v.y * exp2f(v.x - m);
    }
#pragma unroll
    for (int o = G; o < 32; o <<= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const float f = 1.f / (z * (float)G);
#pragma unroll
    for (int k = 0; k < G; ++k) {
      gm[k] = __shfl_sync(0xffffffffu, m, k);
      fac[k] = __shfl_sync(0xffffffffu, f, k);
    }
  }
  for (int i = threadIdx.x; i < n_win; i += DEC_THREADS) {
    float a = 0.f;
#pragma unroll
    for (int h = 0; h < G; ++h) a = fmaf(exp2f(lg[h * cap_words + i] - gm[h]), fac[h], a);
    abar[i] = a;
  }
  __syncthreads();
  unsigned long long best = kNoKey;
  for (int i = threadIdx.x; i < n_own; i += DEC_THREADS) {
    const int r = r_lo + i;
    if (r >= n_obs) break;
    const int lo = max(0, r - rad) - w_lo, hi = min(n_obs, r + rad + 1) - w_lo;
    float v = abar[lo];
    for (int x = lo + 1; x < hi; ++x) v = A.pool_mode == CAKE_POOL_MAX ? fmaxf(v, abar[x]) : v + abar[x];
    if (A.pool_mode != CAKE_POOL_MAX) v /= (float)A.kp;
    float sc = v;
    if (r < n_old) {
      const float o = old[i];
      sc = A.update_mode == CAKE_DECODE_ADD ? o + v : A.update_mode == CAKE_DECODE_MAX ? fmaxf(o, v) : v;
    }
    A.score[base + ord[own + i]] = sc;
    best = min(best, evict_key(sc, r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (lane == 0) red_k[warp] = best;
  __syncthreads();
  if (warp == 0) {
    best = lane < DEC_THREADS / 32 ? red_k[lane] : kNoKey;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
    const int r = 0x7FFFFFFF - (int)(uint32_t)best;
    const uint4 v = make_uint4((uint32_t)(best >> 32), (uint32_t)best, best == kNoKey ? 0u : (uint32_t)ord[r - w_lo], 0u);
    if (csize == 1) { if (lane == 0) x_cand[0] = v; }
    else if (lane < csize) st_remote(&x_cand[crank], (uint32_t)lane, v);
  }
  if (csize > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
  // 5. evict back to the frozen budget: ranks after the evicted one move down by one, its slot
  //    becomes the free one
  best = kNoKey;
  int ev_slot = 0;
  for (int c = 0; c < csize; ++c) {
    const uint4 v = x_cand[c];
    const unsigned long long k = ((unsigned long long)v.x << 32) | v.y;
    if (k < best) { best = k; ev_slot = (int)v.z; }
  }
  if (best == kNoKey || n_obs <= budget) {           // below the budget: the cache would have to grow
    if (crank == 0 && threadIdx.x == 0) atomicCAS(A.status, 0, CAKE_ERR_CAPACITY);
    return;
  }
  const int ev = 0x7FFFFFFF - (int)(uint32_t)best;
  for (int i = max(0, ev - r_lo) + (int)threadIdx.x; i < n_own; i += DEC_THREADS) {
    const int r = r_lo + i;
    A.order[base + r] = r < len ? ord[own + i + 1] : ev_slot;
  }
  if (crank == 0 && threadIdx.x == 0) {
    A.pos[base + ev_slot] = -1;
    A.meta[lid] = make_int4(len, ev_slot, next_pos + 1, budget);
  }
}

// Entries of one (request, layer) in ascending position: positions, scores (window entries 0),
// slots.  One thread per entry, a row of CTAs per head.
__global__ void decode_read_state(const int64_t* __restrict__ dec_off, const float* __restrict__ score,
                                  const int32_t* __restrict__ pos, const int32_t* __restrict__ order,
                                  const int4* __restrict__ meta, int32_t* __restrict__ pos_out,
                                  float* __restrict__ score_out, int32_t* __restrict__ slot_out,
                                  int blk, int Hkv, int Sw) {
  const int g = blockIdx.x;
  const int len = meta[(size_t)blk * Hkv + g].x;
  const int64_t base = dec_off[blk] + (int64_t)g * (len + 1);
  for (int r = blockIdx.y * blockDim.x + threadIdx.x; r < len; r += gridDim.y * blockDim.x) {
    const int s = order[base + r];
    if (pos_out) pos_out[(size_t)g * len + r] = pos[base + s];
    if (slot_out) slot_out[(size_t)g * len + r] = s;
    if (score_out) score_out[(size_t)g * len + r] = r < len - Sw ? score[base + s] : 0.f;
  }
}

template <typename T, int G>
cudaError_t launch_step_cluster_g(dim3 grid, int csize, int cap_words, bool early, size_t smem, cudaStream_t st,
                                  const DecodeArgs& A) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid.x * csize, grid.y, 1);
  cfg.blockDim = dim3(DEC_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, decode_step_cluster_kernel<T, G>, A, csize, cap_words);
}

// Once per device: the kernels' attributes, and whether it holds a cluster of DEC_CLUSTER_WIDE of them all.
template <typename T>
cudaError_t prepare_step_cluster(int device, bool* wide) {
  static PerDeviceOnce attr;
  static bool fits[kOnceDevices];
  if (!attr.need(device)) { *wide = fits[device]; return cudaSuccess; }
  cudaError_t e = cudaSuccess;
  bool all = true;
#define CAKE_DEC_ATTR(GG) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_step_cluster_kernel<T, GG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecSmemMax); \
  all = e == cudaSuccess && cluster_fits(decode_step_cluster_kernel<T, GG>, DEC_CLUSTER_WIDE, DEC_THREADS, kDecSmemMax) && all
  CAKE_DEC_ATTR(1); CAKE_DEC_ATTR(2); CAKE_DEC_ATTR(4); CAKE_DEC_ATTR(8);
#undef CAKE_DEC_ATTR
  if (e != cudaSuccess) return e;
  if (device >= 0 && device < kOnceDevices) fits[device] = all;
  attr.mark(device);
  *wide = all;
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_step_cluster(int G, dim3 grid, int csize, int cap_words, bool early, cudaStream_t st, const DecodeArgs& A) {
  const size_t smem = (size_t)(G + 3) * cap_words * sizeof(float);
  switch (G) {
    case 1: return launch_step_cluster_g<T, 1>(grid, csize, cap_words, early, smem, st, A);
    case 2: return launch_step_cluster_g<T, 2>(grid, csize, cap_words, early, smem, st, A);
    case 4: return launch_step_cluster_g<T, 4>(grid, csize, cap_words, early, smem, st, A);
    case 8: return launch_step_cluster_g<T, 8>(grid, csize, cap_words, early, smem, st, A);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_step(int device, int G, dim3 grid, size_t smem, cudaStream_t st, const DecodeArgs& A) {
  static PerDeviceOnce attr;
  if (attr.need(device)) {
    cudaError_t e = cudaSuccess;
#define CAKE_DEC_ATTR(GG) \
    if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_step_kernel<T, GG>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)
    CAKE_DEC_ATTR(1); CAKE_DEC_ATTR(2); CAKE_DEC_ATTR(4); CAKE_DEC_ATTR(8);
#undef CAKE_DEC_ATTR
    if (e != cudaSuccess) return e;
    attr.mark(device);
  }
  switch (G) {
    case 1: decode_step_kernel<T, 1><<<grid, DEC_THREADS, smem, st>>>(A); break;
    case 2: decode_step_kernel<T, 2><<<grid, DEC_THREADS, smem, st>>>(A); break;
    case 4: decode_step_kernel<T, 4><<<grid, DEC_THREADS, smem, st>>>(A); break;
    case 8: decode_step_kernel<T, 8><<<grid, DEC_THREADS, smem, st>>>(A); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

int32_t launch_decode_begin(cake_ctx* ctx, const LayerPtrs& ptrs, void* k_cache, void* v_cache,
                            int64_t* row_offsets, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int32_t* budget = ctx->d_budget[(ctx->n_evicted - 1) & 1];
  int32_t rc = run_offsets(ctx, 0, c.n_layers, ctx->d_dec_packed_off, nullptr, 1, ctx->d_dec_off, st);
  if (rc != CAKE_OK) return rc;
  // positions in packed order (context scratch), then the decode state and the rows
  rc = run_sorted_positions(ctx, 0, ctx->n_req, 0, c.n_layers, ctx->d_dec_packed_off, ctx->d_pos_packed, 0, st);
  if (rc != CAKE_OK) return rc;
  if (row_offsets)
    CAKE_CUDA_TRY(cudaMemcpyAsync(row_offsets, ctx->d_dec_off, sizeof(int64_t) * (ctx->n_req * c.n_layers + 1),
                                  cudaMemcpyDeviceToDevice, st));
  if (ctx->n_req == 0) return CAKE_OK;
  const dim3 grid(c.n_kv_heads, c.n_layers, ctx->n_req);
  decode_build<<<grid, DEC_THREADS, 0, st>>>(ctx->d_store, ctx->d_req, budget, ctx->d_dec_packed_off,
                                             ctx->d_pos_packed, ctx->d_dec_off, ctx->d_dec_score, ctx->d_dec_pos,
                                             ctx->d_dec_order, ctx->d_dec_meta, c.n_layers, c.n_kv_heads, c.window,
                                             ctx->total_tokens);
  count_launch();
  CAKE_CUDA_TRY(cudaGetLastError());
  return run_gather(ctx, ptrs, ctx->d_dec_packed_off, ctx->d_dec_off, ctx->d_pos_packed, k_cache, v_cache, st);
}

int32_t launch_decode_step(cake_ctx* ctx, int32_t layer, const void* q_new, const void* k_new,
                           const void* v_new, void* k_cache, void* v_cache, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  if (ctx->n_req == 0) return CAKE_OK;
  const int G = c.n_q_heads / c.n_kv_heads;
  DecodeArgs A;
  A.q_new = q_new; A.k_new = k_new; A.v_new = v_new; A.k_cache = k_cache; A.v_cache = v_cache;
  A.dec_off = ctx->d_dec_off; A.score = ctx->d_dec_score; A.pos = ctx->d_dec_pos;
  A.order = ctx->d_dec_order; A.meta = ctx->d_dec_meta; A.status = ctx->d_status;
  A.layer = layer; A.L = c.n_layers; A.Hq = c.n_q_heads; A.Hkv = c.n_kv_heads; A.d = c.head_dim;
  A.Sw = c.window; A.kp = c.pool_kernel; A.pool_mode = c.pool_mode; A.update_mode = ctx->dec_update_mode;
  A.scale2 = 1.4426950408889634f / sqrtf((float)c.head_dim);
  // shared memory: (G + 1) floats per slot, sized for the largest head of the batch up to the
  // 200 KB the kernel may take; larger heads use the context's work area in global memory
  const int64_t limit = (200 * 1024) / ((int64_t)(G + 1) * (int64_t)sizeof(float));
  const int64_t cap = std::min<int64_t>(ctx->dec_max_cap, limit);
  const size_t smem = (size_t)(G + 1) * cap * sizeof(float);
  A.smem_cap = (int)cap;
  A.tmp = ctx->d_dec_tmp; A.reqs = ctx->d_req; A.T = ctx->total_tokens; A.n_req = ctx->n_req;
  const dim3 grid(c.n_kv_heads, ctx->n_req);
  // A head is spread over the fewest CTAs that leave each at most DEC_CTA_ENTRIES entries (one
  // pass of its sixteen warps over 16 key rows each), up to DEC_CLUSTER, or up to DEC_CLUSTER_WIDE
  // while the grid still fits the SMs (at one request of eight heads 64 CTAs would leave half of
  // them idle) and the device holds such a cluster.  Heads whose share does not fit a CTA's shared memory even then, tensors that do
  // not start on a 32-byte boundary, and all heads with CAKE_DECODE_CLUSTER=0, stay on one CTA of
  // the form that reads 8 bytes at a time and can work in global memory.
  const int64_t max_cap = ctx->h_dec_cap[layer];
  const int64_t heads = (int64_t)c.n_kv_heads * ctx->n_req;
  bool wide = false;
  CAKE_CUDA_TRY(c.dtype == CAKE_DTYPE_FP32 ? prepare_step_cluster<float>(ctx->device, &wide)
                                           : prepare_step_cluster<__nv_bfloat16>(ctx->device, &wide));
  const int widest = widest_cluster(wide, DEC_CLUSTER_WIDE);
  int csize = 1;
  while (max_cap > (int64_t)csize * DEC_CTA_ENTRIES && csize * 2 <= widest &&
         (csize < DEC_CLUSTER || (csize < DEC_CLUSTER_WIDE && heads * csize * 2 <= ctx->n_sm)))
    csize *= 2;
  const int64_t words = (max_cap + csize - 1) / csize + 2 * (c.pool_kernel / 2) + 2;
  const bool aligned = (((uintptr_t)q_new | (uintptr_t)k_new | (uintptr_t)v_new | (uintptr_t)k_cache | (uintptr_t)v_cache) & 31) == 0;
  const char* env = getenv("CAKE_DECODE_CLUSTER");
  const bool use_cluster = aligned && (size_t)(G + 3) * words * sizeof(float) <= kDecSmemMax && !(env && env[0] == '0');
  // A step may start while the kernel before it in the stream still runs, read its layer's state and
  // bring the layer's keys towards the SMs, and then wait.  That state was last written by the same
  // layer's previous step (or by the set-up of the cache).  A step lets its successor start only after its
  // own predecessor in the stream has finished, so what was enqueued on this stream before the step before
  // this one is complete by then.  Hence only when the step before this one is another layer's on this
  // stream, and this layer's own one was on this stream too (a step on another stream may have been
  // ordered before this one by an event that the launch waits for, or may not: no early start).  A captured
  // graph runs as a whole behind everything before it, so steps that ran earlier are complete when it
  // starts; steps beside a replayed graph cannot tell what it has stepped.
  const StepPlace here = step_place(st);
  auto same = [](const StepPlace& a, const StepPlace& b) { return a.stream != 0 && a.stream == b.stream && a.capture == b.capture; };
  const StepPlace& own = ctx->dec_place[layer];
  const bool early = ctx->dec_last_layer >= 0 && ctx->dec_last_layer != layer && same(ctx->dec_last, here) &&
                     (here.capture ? own.capture != here.capture || same(own, here) : !ctx->dec_captured && same(own, here));
  cudaError_t e;
  if (use_cluster)
    e = c.dtype == CAKE_DTYPE_FP32 ? launch_step_cluster<float>(G, grid, csize, (int)words, early, st, A)
                                   : launch_step_cluster<__nv_bfloat16>(G, grid, csize, (int)words, early, st, A);
  else
    e = c.dtype == CAKE_DTYPE_FP32 ? launch_step<float>(ctx->device, G, grid, smem, st, A)
                                   : launch_step<__nv_bfloat16>(ctx->device, G, grid, smem, st, A);
  count_launch();
  ctx->dec_last_layer = use_cluster && e == cudaSuccess ? layer : -1;
  ctx->dec_last = ctx->dec_place[layer] = here;
  ctx->dec_captured = ctx->dec_captured || here.capture != 0;
  return cuda_status(e);
}

int32_t launch_decode_read(cake_ctx* ctx, int32_t req, int32_t layer, int32_t* positions, float* scores,
                           int32_t* slots, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const dim3 grid(c.n_kv_heads, (unsigned)std::min<int64_t>(64, (ctx->h_dec_cap[layer] + 255) / 256));
  decode_read_state<<<grid, 256, 0, st>>>(ctx->d_dec_off, ctx->d_dec_score, ctx->d_dec_pos,
                                                  ctx->d_dec_order, ctx->d_dec_meta, positions, scores, slots,
                                                  req * c.n_layers + layer, c.n_kv_heads, c.window);
  count_launch();
  return cuda_status(cudaGetLastError());
}

}  // namespace cake
