// Window-score kernels, plain fp32 SIMT version.
//
// Serves fp32 inputs (and any shape the tensor-core path does not take).  Per layer:
//   scores_simt     base-2 logits of every (request, KV head), tile by tile: kept in a work area of the
//                   context for the second kernel, and reduced to row statistics (maximum, sum); the CTA
//                   that finishes a (request, head) merges them into the base-2 log-sum-exp of every
//                   window row over its visible keys (softmax denominator, Section 2 Eq. 2)
//   colstats_simt   column statistics of the normalised probabilities of the non-window keys -> raw
//                   indicator (Eq. 11), per-head sums for the dispersion (Eq. 4) and the shift (Eq. 5)
// The logits are computed once: writing and reading one costs 8 bytes of (mostly L2) traffic, computing
// it again d = 128 FMAs, three times as long even from DRAM.  Where the logits of the batch do not fit
// the work area, or the caller supplies the denominators, the second kernel takes them slice by slice.
#include "cake_internal.cuh"

#include <math_constants.h>

#include <algorithm>

namespace cake {
namespace {

constexpr int NT = kSimtThreads;    // 256 threads
constexpr int CK = 32;              // elements of a row staged at a time

// Four consecutive elements of a staged row.
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xFFFF0000u));
}
// 16 bytes on their way to shared memory; zeros where `in` is false.
__device__ __forceinline__ void copy_async16(void* dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0)
               : "memory");
}

struct ScoreArgs {
  const ScoreUnit* units;
  float2* rowpart;         // [unit][H_kv][rows] (max, sum), or null: logits only
  float* lse2;             // [req][H_kv][rows]
  uint32_t* arrivals;      // [req * H_kv + g] finished units (zero at rest)
  float* scores;           // [unit - u0][H_kv][rows][unit_keys], or null: row statistics only
  int u0, unit_keys, Hq, Hkv, Sw, d;
  int64_t T_tokens;
  float scale2;
};

// TY groups of 8 rows x TX groups of KPT keys; a thread owns 8 rows x KPT keys (rows ty, ty + TY, ... and keys
// tx, tx + TX, ..., so that a warp's reads of either lie in different banks).
// 16 row groups: 128 rows x 64 keys; fewer rows: 128 keys.
template <typename T, int TY> struct Shape {
  static constexpr int TX = NT / TY;
  static constexpr int KPT = TY == 16 ? 4 : TY == 8 ? 4 : TY == 4 ? 2 : 1;
  static constexpr int TK = TX * KPT;
  static constexpr int CS = CK + 16 / (int)sizeof(T);   // padded stride: reads of consecutive rows hit all banks
  static constexpr int STAGE = (TY * 8 + TK) * CS;      // elements
  static constexpr size_t kSmem = 2 * (size_t)STAGE * sizeof(T) + 8 * NT * sizeof(float2);
};

// One CTA per (unit, KV head).  Bound: issue slots (61 % busy) and the last wave: 393 M FMAs per layer at
// 128 rows, d = 128 and 4 heads of 6K keys are 11 us of the FMA pipe, which is 45 % busy in the 38 us that it
// takes; 376 CTAs for 444 places leave an SM with two or three.  The next piece of the rows is copied to shared memory while a piece is multiplied, and
// three CTAs share an SM.  (One CTA per SM that staged whole rows of 134 KB before it multiplied took
// 56 us there, and its second pass over the keys another 45.)
template <typename T, int TY>
__global__ void __launch_bounds__(NT, 3)
scores_simt(const T* __restrict__ q_win, const T* __restrict__ k, const ScoreArgs A) {
  using Sh = Shape<T, TY>;
  constexpr int TX = Sh::TX, KPT = Sh::KPT, TK = Sh::TK, R8 = TY * 8, CS = Sh::CS;
  constexpr int E = 16 / (int)sizeof(T), VPR = CK / E;          // 16-byte vectors of a staged row
  extern __shared__ __align__(16) uint8_t smem_raw[];
  T* const smem = reinterpret_cast<T*>(smem_raw);
  __shared__ float2 s_red[NT / 32][8];
  __shared__ int s_last;
  const int G = A.Hq / A.Hkv, rows = G * A.Sw, d = A.d;
  const int g = blockIdx.y, unit = A.u0 + (int)blockIdx.x;
  const ScoreUnit u = A.units[unit];
  const int tid = threadIdx.x, ty = tid / TX, tx = tid % TX;
  const T* qb = q_win + ((size_t)u.req * A.Hq + (size_t)g * G) * A.Sw * d;
  const T* kb = k + ((size_t)g * A.T_tokens + u.cu + u.key0) * d;
  const int nch = d / CK, ntile = (u.nkeys + TK - 1) / TK, steps = nch * ntile;
  auto fetch = [&](int st) {
    const int t0 = st / nch * TK, c0 = st % nch * CK;
    T* qs = smem + (st & 1) * Sh::STAGE;
    T* ks = qs + R8 * CS;
#pragma unroll
    for (int v = tid; v < R8 * VPR; v += NT) {
      const int row = v / VPR, x = v % VPR * E;
      copy_async16(qs + row * CS + x, qb + (size_t)min(row, rows - 1) * d + c0 + x, row < rows);
    }
#pragma unroll
    for (int v = tid; v < TK * VPR; v += NT) {
      const int key = v / VPR, x = v % VPR * E;
      copy_async16(ks + key * CS + x, kb + (size_t)min(t0 + key, u.nkeys - 1) * d + c0 + x, t0 + key < u.nkeys);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // running maximum and sum of this thread's rows: in shared memory, they are needed once per tile
  float2* const mz = reinterpret_cast<float2*>(smem_raw + 2 * (size_t)Sh::STAGE * sizeof(T)) + tid;
#pragma unroll
  for (int r = 0; r < 8; ++r) mz[r * NT] = make_float2(-CUDART_INF_F, 0.f);
  float acc[8][KPT];
  // up to here nothing was read or written that the kernel before this one, which may still run, has to do with
  asm volatile("griddepcontrol.wait;" ::: "memory");
  fetch(0);
#pragma unroll 1
  for (int st = 0; st < steps; ++st) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                  // this piece has landed, and the other buffer's readers are done
    if (st + 1 < steps) fetch(st + 1);
    const T* qs = smem + (st & 1) * Sh::STAGE + ty * CS;
    const T* ks = smem + (st & 1) * Sh::STAGE + (R8 + tx) * CS;
    if (st % nch == 0)
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < KPT; ++c) acc[r][c] = 0.f;
#pragma unroll 4
    for (int c = 0; c < CK; c += 4) {
      float4 kf[KPT];
#pragma unroll
      for (int x = 0; x < KPT; ++x) kf[x] = load4(ks + TX * x * CS + c);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 qf = load4(qs + r * TY * CS + c);
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          acc[r][x] = fmaf(qf.x, kf[x].x, acc[r][x]);
          acc[r][x] = fmaf(qf.y, kf[x].y, acc[r][x]);
          acc[r][x] = fmaf(qf.z, kf[x].z, acc[r][x]);
          acc[r][x] = fmaf(qf.w, kf[x].w, acc[r][x]);
        }
      }
    }
    if (st % nch != nch - 1) continue;
    // the tile's logits: out, and into this thread's running maximum and sum of every row
    const int t0 = st / nch * TK;
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int x = 0; x < KPT; ++x) acc[r][x] *= A.scale2;
    if (A.scores) {
      float* out = A.scores + (((size_t)blockIdx.x * A.Hkv + g) * rows + ty) * A.unit_keys + t0 + tx;
#pragma unroll
      for (int r = 0; r < 8; ++r, out += TY * A.unit_keys)
        if (r * TY + ty < rows)
#pragma unroll
          for (int x = 0; x < KPT; ++x)
            if (t0 + tx + TX * x < u.nkeys) out[TX * x] = acc[r][x];
    }
    if (!A.rowpart) continue;
    if (t0 + TK > u.nkeys || u.key0 + t0 + TK > u.n) {          // ragged end, or keys that some rows do not see
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int last = u.n + (r * TY + ty) % A.Sw;   // last key the row may see
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const int key = t0 + tx + TX * x;
          if (key >= u.nkeys || u.key0 + key > last) acc[r][x] = -CUDART_INF_F;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float mx = acc[r][0];
#pragma unroll
      for (int x = 1; x < KPT; ++x) mx = fmaxf(mx, acc[r][x]);
      if (mx == -CUDART_INF_F) continue;
      const float2 old = mz[r * NT];
      const float mn = fmaxf(old.x, mx);
      float e = old.y > 0.f ? old.y * exp2f(old.x - mn) : 0.f;
#pragma unroll
      for (int x = 0; x < KPT; ++x) e += exp2f(acc[r][x] - mn);
      mz[r * NT] = make_float2(mn, e);
    }
  }
  // The column pass may take its places; it waits for this kernel's end before it reads.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!A.rowpart) return;
  // over the threads of a row group, in a fixed order: maxima, then sums against them
  const int lane = tid & 31, warp = tid >> 5;
  float m[8], z[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float2 own = mz[r * NT];
    float mx = own.x;
#pragma unroll
    for (int o = 1; o < (TX < 32 ? TX : 32); o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float e = own.y > 0.f ? own.y * exp2f(own.x - mx) : 0.f;
#pragma unroll
    for (int o = 1; o < (TX < 32 ? TX : 32); o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    m[r] = mx;
    z[r] = e;
    if (TX > 32 && lane == 0) s_red[warp][r] = make_float2(mx, e);
  }
  auto merge = [](float2 a, float2 b) {
    const float mn = fmaxf(a.x, b.x);
    if (mn == -CUDART_INF_F) return a;
    return make_float2(mn, a.y * exp2f(a.x - mn) + b.y * exp2f(b.x - mn));
  };
  if (TX > 32) __syncthreads();
  float2* part = A.rowpart + ((size_t)unit * A.Hkv + g) * rows;
  if (tx == 0) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float2 a = make_float2(m[r], z[r]);
      if (TX > 32)
        for (int w = 1; w < TX / 32; ++w) a = merge(a, s_red[warp + w][r]);
      if (r * TY + ty < rows) part[r * TY + ty] = a;
    }
  }
  // the CTA that finishes the (request, head) merges the units' rows, two threads per row
  const int pair = u.req * A.Hkv + g;
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    s_last = atomicAdd(&A.arrivals[pair], 1u) + 1u == (uint32_t)u.nunits ? 1 : 0;
    if (s_last) A.arrivals[pair] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int row = tid >> 1, half = (u.nunits + 1) / 2;
  const int a0 = u.unit0 + (tid & 1 ? half : 0), a1 = u.unit0 + (tid & 1 ? u.nunits : half);
  float2 acc2 = make_float2(-CUDART_INF_F, 0.f);
  if (row < rows) {
    for (int i = a0; i < a1; i += 16) {
      float2 p[16];
#pragma unroll
      for (int x = 0; x < 16; ++x)
        p[x] = i + x < a1 ? __ldcg(&A.rowpart[((size_t)(i + x) * A.Hkv + g) * rows + row]) : make_float2(-CUDART_INF_F, 0.f);
      float mn = acc2.x;
#pragma unroll
      for (int x = 0; x < 16; ++x) mn = fmaxf(mn, p[x].x);
      if (mn == -CUDART_INF_F) continue;
      float e = acc2.y * exp2f(acc2.x - mn);
#pragma unroll
      for (int x = 0; x < 16; ++x) e = fmaf(p[x].y, exp2f(p[x].x - mn), e);
      acc2 = make_float2(mn, e);
    }
  }
  const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, acc2.x, 1), __shfl_xor_sync(0xffffffffu, acc2.y, 1));
  acc2 = merge(acc2, other);
  if (!(tid & 1) && row < rows) A.lse2[(size_t)pair * rows + row] = acc2.x + log2f(acc2.y);
}

__global__ void lse_to_base2(const float* __restrict__ lse, float* __restrict__ lse2, int64_t count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) lse2[i] = lse[i] * 1.4426950408889634f;
}

__device__ inline float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct ColArgs {
  const ScoreUnit* units;
  const float* lse2;
  const float* scores;
  float* raw;
  float* colpart;
  int u0, unit_keys, Hq, Hkv, Sw;
  int64_t T_tokens;
  float gamma;
  int ddof, ind_mode;
};

// One CTA per (unit, KV head): 64 keys at a time, a lane per key, and four quarters of the window rows
// on two warps each.  Bound: the latency of the loads: 14 us for 4 heads of 6K keys and 128 rows at 30 % of the
// issue slots and 7 % of the special-function unit, with two window rows in flight.  A thread now has 16 logits in
// flight (8 where a KV head has one query head), as many as the registers of three CTAs per SM allow: eight layers
// take 402 us with two rows at a time and 381 so, where the next kernel starts early; where it does not, 432 and 429.
// With more than four query heads per KV head these registers do not hold a thread's sums and logits, and it is two CTAs
// per SM: eight layers of 6K keys with 16 heads on 2 take 344 us so and 363 with three, which spilled; 32 on 4 400 and 404.
constexpr int COL_KEYS = 64;
template <int GM>          // query heads per KV head, at most
__global__ void __launch_bounds__(NT, GM > 4 ? 2 : 3)
colstats_simt(const ColArgs A) {
  __shared__ float s_lse[kMaxRows];
  __shared__ float s_part[4][2 + 2 * GM][COL_KEYS];
  __shared__ float s_red[NT / 32][2 * GM];
  constexpr int COL_BATCH = GM <= 2 ? 8 : 16 / GM;        // window rows of a thread whose loads are in flight together
  const int G = A.Hq / A.Hkv, rows = G * A.Sw;
  const int g = blockIdx.y, unit = A.u0 + (int)blockIdx.x;
  const ScoreUnit u = A.units[unit];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // the logits and the denominators come from the kernel before this one, which may still run
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int quarter = warp >> 1, key_l = (warp & 1) * 32 + lane;
  const float* sc = A.scores + ((size_t)blockIdx.x * A.Hkv + g) * rows * A.unit_keys;
  for (int r = tid; r < rows; r += NT) s_lse[r] = A.lse2[((size_t)u.req * A.Hkv + g) * rows + r];
  float hs[GM], vacc[GM];
#pragma unroll
  for (int h = 0; h < GM; ++h) { hs[h] = 0.f; vacc[h] = 0.f; }
  const int nkeys = min(u.nkeys, u.n - u.key0);       // only non-window keys
  const float inv_sw = 1.f / (float)A.Sw, inv_g = 1.f / (float)G;
  const float bessel = A.ddof ? (float)A.Sw / (float)(A.Sw - 1) : 1.f;
  __syncthreads();
  for (int k0 = 0; k0 < nkeys; k0 += COL_KEYS) {
    const bool valid = k0 + key_l < nkeys;
    const float* col = sc + (valid ? k0 + key_l : 0);
    float s1[GM], s2[GM], a1 = 0.f, a2 = 0.f;
#pragma unroll
    for (int h = 0; h < GM; ++h) { s1[h] = 0.f; s2[h] = 0.f; }
    for (int i0 = quarter; i0 < A.Sw; i0 += 4 * COL_BATCH) {
      float x[COL_BATCH][GM];
#pragma unroll
      for (int e = 0; e < COL_BATCH; ++e)
#pragma unroll
        for (int h = 0; h < GM; ++h)
          x[e][h] = h < G && i0 + 4 * e < A.Sw ? __ldcg(&col[(size_t)(h * A.Sw + i0 + 4 * e) * A.unit_keys]) : 0.f;
#pragma unroll
      for (int e = 0; e < COL_BATCH; ++e) {
        const int i = i0 + 4 * e;
        if (i >= A.Sw) break;
        float a = 0.f;
#pragma unroll
        for (int h = 0; h < GM; ++h) {
          if (h < G) {
            const float v = x[e][h] - s_lse[h * A.Sw + i], p = exp2f(v);
            hs[h] = fmaf(valid ? p : 0.f, v, hs[h]);
            s1[h] += p;
            s2[h] = fmaf(p, p, s2[h]);
            a += p;
          }
        }
        a *= inv_g;
        a1 += a;
        a2 = fmaf(a, a, a2);
      }
    }
    s_part[quarter][0][key_l] = a1;
    s_part[quarter][1][key_l] = a2;
#pragma unroll
    for (int h = 0; h < GM; ++h) {
      if (h < G) { s_part[quarter][2 + 2 * h][key_l] = s1[h]; s_part[quarter][3 + 2 * h][key_l] = s2[h]; }
    }
    __syncthreads();
    if (quarter == 0 && valid) {
      auto sum = [&](int x) { return (s_part[0][x][key_l] + s_part[1][x][key_l]) + (s_part[2][x][key_l] + s_part[3][x][key_l]); };
      const float mean = sum(0) * inv_sw;
      const float var = fmaxf(sum(1) * inv_sw - mean * mean, 0.f) * bessel;
      A.raw[(size_t)g * A.T_tokens + u.cu + u.key0 + k0 + key_l] = combine_indicator(A.ind_mode, A.gamma, mean, var, (float)A.Sw);
#pragma unroll
      for (int h = 0; h < GM; ++h) {
        if (h < G) {
          const float mh = sum(2 + 2 * h) * inv_sw;
          vacc[h] += fmaxf(sum(3 + 2 * h) * inv_sw - mh * mh, 0.f) * bessel;
        }
      }
    }
    __syncthreads();
  }
  // fixed-order block reduction of hs / vacc: warp shuffle tree, then over the warps
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    const float a = warp_sum(hs[h]);
    const float b = warp_sum(vacc[h]);
    if (lane == 0) { s_red[warp][h] = a; s_red[warp][GM + h] = b; }
  }
  __syncthreads();
  if (tid < 2 * G) {
    const int h = tid >> 1, which = tid & 1;
    float acc = 0.f;
    for (int w = 0; w < NT / 32; ++w) acc += s_red[w][which * GM + h];
    A.colpart[(((size_t)unit * A.Hkv + g) * G + h) * 2 + which] = acc;
  }
}

// A launch whose CTAs may take their places while the kernel before it ends (both kernels wait for that end before
// they touch what others do).  Without it a layer's two kernels and the next layer's each stood 2 to 3 us apart: eight
// layers of 6K keys 429 -> 381 us, four of 512 keys 100 -> 82.  scores_simt lets the column pass in once its logits are
// out; from its start on it is slower (389 us), since the waiting CTAs hold registers.
template <typename... Params, typename... Args>
cudaError_t launch_early(void (*kernel)(Params...), dim3 grid, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T, int TY>
cudaError_t launch_scores(int device, dim3 grid, cudaStream_t st, const void* q, const void* k, const ScoreArgs& A) {
  static PerDeviceOnce attr;
  if (attr.need(device)) {
    const cudaError_t e = cudaFuncSetAttribute(scores_simt<T, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Shape<T, TY>::kSmem);
    if (e != cudaSuccess) return e;
    attr.mark(device);
  }
  const cudaError_t e = launch_early(scores_simt<T, TY>, grid, Shape<T, TY>::kSmem, st, (const T*)q, (const T*)k, A);
  count_launch();
  return e;
}

template <typename T>
int32_t run(cake_ctx* ctx, int32_t layer, const void* q_win, const void* k, const float* lse,
            cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int rows = ctx->rows, G = c.n_q_heads / c.n_kv_heads;
  ScoreArgs A;
  A.units = ctx->d_units; A.lse2 = ctx->d_lse2; A.arrivals = ctx->d_simt_arrivals;
  A.unit_keys = ctx->unit_keys; A.Hq = c.n_q_heads; A.Hkv = c.n_kv_heads; A.Sw = c.window; A.d = c.head_dim;
  A.T_tokens = ctx->total_tokens;
  A.scale2 = 1.4426950408889634f / sqrtf((float)c.head_dim);
  auto scores = [&](int u0, int n, bool rowstats, bool store) {
    A.u0 = u0;
    A.rowpart = rowstats ? ctx->d_rowpart : nullptr;
    A.scores = store ? ctx->d_scores : nullptr;
    const dim3 grid(n, c.n_kv_heads);
    // the fewest groups of 8 rows that hold the window rows
    if (rows > 64) return launch_scores<T, 16>(ctx->device, grid, st, q_win, k, A);
    if (rows > 32) return launch_scores<T, 8>(ctx->device, grid, st, q_win, k, A);
    if (rows > 16) return launch_scores<T, 4>(ctx->device, grid, st, q_win, k, A);
    return launch_scores<T, 2>(ctx->device, grid, st, q_win, k, A);
  };
  // units whose logits fit the work area together
  const int64_t per_unit = (int64_t)c.n_kv_heads * rows * ctx->unit_keys;
  const int slice = (int)std::min<int64_t>(ctx->n_units, ctx->scores_elems / per_unit);
  const bool whole = slice == ctx->n_units;
  int sp = prof_begin(ctx, CAKE_PROF_SCORE, st);
  if (lse) {
    const int64_t n_lse = (int64_t)ctx->n_req * c.n_q_heads * c.window;
    lse_to_base2<<<(unsigned)((n_lse + 255) / 256), 256, 0, st>>>(lse, ctx->d_lse2, n_lse);
    count_launch();
  } else {
    CAKE_CUDA_TRY(scores(0, ctx->n_units, true, whole));
  }
  prof_end(ctx, sp, st);
  sp = prof_begin(ctx, CAKE_PROF_SCORE, st);
  ColArgs B;
  B.units = ctx->d_units; B.lse2 = ctx->d_lse2; B.scores = ctx->d_scores;
  B.raw = ctx->d_raw[layer % ctx->score_depth]; B.colpart = ctx->d_colpart[layer % ctx->score_depth];
  B.unit_keys = ctx->unit_keys; B.Hq = c.n_q_heads; B.Hkv = c.n_kv_heads; B.Sw = c.window;
  B.T_tokens = ctx->total_tokens; B.gamma = c.gamma; B.ddof = c.var_ddof; B.ind_mode = c.indicator_mode;
  for (int u0 = 0; u0 < ctx->n_units; u0 += slice) {
    const int n = std::min(slice, ctx->n_units - u0);
    if (lse || !whole) CAKE_CUDA_TRY(scores(u0, n, false, true));
    B.u0 = u0;
    const dim3 grid(n, c.n_kv_heads);
    CAKE_CUDA_TRY(launch_early(G == 1 ? colstats_simt<1> : G == 2 ? colstats_simt<2> : G <= 4 ? colstats_simt<4> : colstats_simt<8>, grid, 0, st, B));
    count_launch();
  }
  prof_end(ctx, sp, st);
  return cuda_status(cudaGetLastError());
}

}  // namespace

int32_t simt_tile_keys(int rows) { return rows > 64 ? Shape<float, 16>::TK : rows > 32 ? Shape<float, 8>::TK : rows > 16 ? Shape<float, 4>::TK : Shape<float, 2>::TK; }

int32_t launch_score_simt(cake_ctx* ctx, int32_t layer, const void* q_win, const void* k,
                          const float* lse, cudaStream_t st) {
  if (ctx->n_units == 0) return CAKE_OK;
  if (ctx->cfg.dtype == CAKE_DTYPE_FP32) return run<float>(ctx, layer, q_win, k, lse, st);
  return run<__nv_bfloat16>(ctx, layer, q_win, k, lse, st);
}

}  // namespace cake
