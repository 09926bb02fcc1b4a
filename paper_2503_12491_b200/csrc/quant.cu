// Quantised gather-compaction: the retained K/V rows (Eq. 12) written as asymmetric 4-bit codes,
// keys per channel and values per token -- the "KIVI-INT4 with CAKE" combination of the paper's
// appendix "Comparison and Compatibility with Quantization Methods".
//
// A group of `group` values shares zero = min and scale = (max - min) / 15 (scale = 1 when
// max = min); code = clamp(rint((x - zero) / scale), 0, 15), all in IEEE fp32 (round to nearest
// even), two codes per byte (the even-numbered channel in the low nibble).
//   values: a group is `group` consecutive channels of one retained row;
//   keys:   a group is one channel over `group` consecutive retained rows of one (request, layer,
//           head) in packed order (ascending position, window last); the last group of a head
//           may be shorter.
#include "cake_internal.cuh"

#include <math_constants.h>

namespace cake {
namespace {

// Two fp32 values in one register pair and the packed arithmetic on them (one issue for two results).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ uint32_t code4(float x, float zero, float scale) {
  const float q = rintf(__fdiv_rn(__fsub_rn(x, zero), scale));
  return (uint32_t)fminf(fmaxf(q, 0.f), 15.f);
}
__device__ __forceinline__ float scale_of(float mn, float mx) {
  return mx > mn ? __fdiv_rn(__fsub_rn(mx, mn), 15.f) : 1.f;
}

// Eight consecutive channels of a row as they lie in memory (kVec: on a 16-byte boundary, in vector
// loads).
template <typename T, bool kVec> struct Oct;
template <bool kVec> struct Oct<float, kVec> {
  float x[8];
  __device__ __forceinline__ void load(const float* p) {
    if constexpr (kVec) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
      x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = p[e];
    }
  }
  __device__ __forceinline__ void values(int half, float (&v)[4]) const {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = x[4 * half + e];
  }
};
template <bool kVec> struct Oct<__nv_bfloat16, kVec> {
  uint32_t w[4];
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    if constexpr (kVec) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(p));
      w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
    } else {
      const uint16_t* q = reinterpret_cast<const uint16_t*>(p);
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = q[2 * i] | (uint32_t)q[2 * i + 1] << 16;
    }
  }
  __device__ __forceinline__ void values(int half, float (&v)[4]) const {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      v[2 * i] = __uint_as_float(w[2 * half + i] << 16);
      v[2 * i + 1] = __uint_as_float(w[2 * half + i] & 0xFFFF0000u);
    }
  }
  __device__ __forceinline__ __nv_bfloat162 pair(int i) const { return *reinterpret_cast<const __nv_bfloat162*>(&w[i]); }
};

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Codes of four values in bits 0..15, from -zero, 1 / scale (rounded to nearest) and -scale.  A code is
// the IEEE quotient (x - zero) / scale rounded half to even.  About 0.2 % of bf16 inputs lie exactly
// half-way, so the quotient has to be the correctly rounded one: the product with the reciprocal,
// corrected once by its exact remainder (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", 1990).  The rounding to an integer is an addition of 1.5 * 2^23.
// `odd` is set when the four are not all in 0..15: an operand is not finite, or the reciprocal is not a
// number because the scale is out of the range in which the remainder is exact (`safe_rcp`).
// (Testing for "near one half" and dividing there cost more than this: 22 % of the warps' rows have one.)
__device__ __forceinline__ uint32_t fast_codes(const float (&x)[4], const f32x2 (&nzero)[2], const f32x2 (&rcp)[2],
                                               const f32x2 (&nscale)[2], bool& odd) {
  constexpr float kMagic = 12582912.f;
  const f32x2 up = pack2(kMagic, kMagic), minus = pack2(-1.f, -1.f);
  float n[4];                                        // minus the codes
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const f32x2 dlt = add2(pack2(x[2 * p], x[2 * p + 1]), nzero[p]);
    const f32x2 q = mul2(dlt, rcp[p]);
    unpack2(fma2(add2(fma2(fma2(q, nscale[p], dlt), rcp[p], q), up), minus, up), n[2 * p], n[2 * p + 1]);
  }
  const float v = __fmaf_rn(__fmaf_rn(n[3], 16.f, n[2]), 256.f, __fmaf_rn(n[1], 16.f, n[0]));
  odd = !(v <= 0.f && v >= -65535.f);
  return __float_as_uint(__fsub_rn(kMagic, v)) & 0xFFFFu;
}
__device__ __forceinline__ float safe_rcp(float scale) {
  return scale >= 0x1p-90f && scale <= 0x1p90f ? __frcp_rn(scale) : CUDART_NAN_F;
}
__device__ __noinline__ uint32_t exact_codes(float x0, float x1, float x2, float x3, float z0, float z1, float z2, float z3,
                                             float s0, float s1, float s2, float s3) {
  return code4(x0, z0, s0) | code4(x1, z1, s1) << 4 | code4(x2, z2, s2) << 8 | code4(x3, z3, s3) << 12;
}

template <bool kVec> __device__ __forceinline__ void put_codes(uint8_t* p, uint32_t c) {
  if constexpr (kVec) {
    *reinterpret_cast<uint32_t*>(p) = c;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = (uint8_t)(c >> (8 * i));
  }
}

// Ranges.  A value that is not a number does not take part.  For bf16 inputs the bounds are exact in
// bf16: two channels at a time, and (min, -max) of a group of channels travel as one register.
template <typename T> struct Channels;               // range of each of a lane's eight channels over rows
template <> struct Channels<float> {
  float mn[8], mx[8];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int e = 0; e < 8; ++e) { mn[e] = CUDART_INF_F; mx[e] = -CUDART_INF_F; }
  }
  template <bool V> __device__ __forceinline__ void add(const Oct<float, V>& o) {
#pragma unroll
    for (int e = 0; e < 8; ++e) { mn[e] = fminf(mn[e], o.x[e]); mx[e] = fmaxf(mx[e], o.x[e]); }
  }
  __device__ __forceinline__ void get(float (&a)[8], float (&b)[8]) const {
#pragma unroll
    for (int e = 0; e < 8; ++e) { a[e] = mn[e]; b[e] = mx[e]; }
  }
};
template <> struct Channels<__nv_bfloat16> {
  __nv_bfloat162 mn[4], mx[4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mn[i] = __floats2bfloat162_rn(CUDART_INF_F, CUDART_INF_F);
      mx[i] = __floats2bfloat162_rn(-CUDART_INF_F, -CUDART_INF_F);
    }
  }
  template <bool V> __device__ __forceinline__ void add(const Oct<__nv_bfloat16, V>& o) {
#pragma unroll
    for (int i = 0; i < 4; ++i) { mn[i] = __hmin2(mn[i], o.pair(i)); mx[i] = __hmax2(mx[i], o.pair(i)); }
  }
  __device__ __forceinline__ void get(float (&a)[8], float (&b)[8]) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[2 * i] = __low2float(mn[i]); a[2 * i + 1] = __high2float(mn[i]);
      b[2 * i] = __low2float(mx[i]); b[2 * i + 1] = __high2float(mx[i]);
    }
  }
};
template <typename T> struct MinMax;                 // range over channels of one row
template <> struct MinMax<float> {
  float mn, mx;
  template <bool V> __device__ __forceinline__ void set(const Oct<float, V>& o) {
    mn = CUDART_INF_F;
    mx = -CUDART_INF_F;
#pragma unroll
    for (int e = 0; e < 8; ++e) { mn = fminf(mn, o.x[e]); mx = fmaxf(mx, o.x[e]); }
  }
  __device__ __forceinline__ void get(float& a, float& b) const { a = mn; b = mx; }
  __device__ __forceinline__ MinMax moved(int o) const {
    return MinMax{__shfl_xor_sync(0xffffffffu, mn, o), __shfl_xor_sync(0xffffffffu, mx, o)};
  }
  __device__ __forceinline__ void merge(const MinMax& b) { mn = fminf(mn, b.mn); mx = fmaxf(mx, b.mx); }
};
template <> struct MinMax<__nv_bfloat16> {
  __nv_bfloat162 v;
  template <bool V> __device__ __forceinline__ void set(const Oct<__nv_bfloat16, V>& o) {
    const __nv_bfloat162 inf = __floats2bfloat162_rn(CUDART_INF_F, CUDART_INF_F);
    const __nv_bfloat162 a = __hmin2(__hmin2(__hmin2(inf, o.pair(0)), o.pair(1)), __hmin2(o.pair(2), o.pair(3)));
    const __nv_bfloat162 b = __hneg2(__hmax2(__hmax2(__hmax2(__hneg2(inf), o.pair(0)), o.pair(1)), __hmax2(o.pair(2), o.pair(3))));
    v = __hmin2(__lows2bfloat162(a, b), __highs2bfloat162(a, b));
  }
  __device__ __forceinline__ void get(float& a, float& b) const { a = __low2float(v); b = -__high2float(v); }
  __device__ __forceinline__ MinMax moved(int o) const { return MinMax{__shfl_xor_sync(0xffffffffu, v, o)}; }
  __device__ __forceinline__ void merge(const MinMax& b) { v = __hmin2(v, b.v); }
};

constexpr int QU_WARPS = 4;

// One warp per 32 packed rows of a key group (group / 32 warps of a CTA share a group and exchange
// their ranges): the keys' ranges, their codes (the second read of the rows hits L1), then the
// values of the same rows.  A lane owns eight channels of a row (D / 8 lanes per row, 2 or 4 rows per
// pass, NB passes of loads in flight).  The values' ranges are reduced and scattered over the lanes,
// so that each lane computes one scale (an IEEE division) for one row and group instead of all
// of them for every row.
//
// Bound: the latency of a warp's chain (positions, rows, ranges, rows again, codes) at the 20 warps that
// 80 registers leave an SM; neither issue slots (54 % busy; ALU and FMA pipes 36 % each) nor DRAM (34 %) are
// full: 60 us for 262 K rows, 190 us for 1.05 M (GQA 32/8, d = 128, group 32).  One warp per
// row with its own search for the row's block and a division near every half-integer, and a CTA per
// key group, took 562 + 445 us for 1.05 M rows.  Keeping the 32 key rows in
// registers instead of reading them twice halved the warps in flight and took 1.2 times as long.
template <typename T, int D, int GW, bool kVec>
__global__ void __launch_bounds__(QU_WARPS * 32, sizeof(T) == 2 ? 6 : 5)
quant_rows(const LayerPtrs ptrs, const int64_t* __restrict__ row_off, const int64_t* __restrict__ key_off,
           const int32_t* __restrict__ budget, const int32_t* __restrict__ pos_packed, const ReqInfo* __restrict__ reqs,
           uint8_t* __restrict__ k_codes, float* __restrict__ k_scale, float* __restrict__ k_zero,
           uint8_t* __restrict__ v_codes, float* __restrict__ v_scale, float* __restrict__ v_zero, int n_req, int L, int Hkv,
           int Sw, int64_t T_tokens) {
  constexpr int GROUP = GW * 32;
  constexpr int LPR = D / 8, RPP = 32 / LPR, NIT = 32 / RPP;    // lanes per row, rows per pass, passes
  constexpr int NB = 4;                                         // passes whose loads are in flight together
  constexpr uint32_t kAll = 0xffffffffu;
  __shared__ float s_mn[QU_WARPS][D], s_mx[QU_WARPS][D];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane / LPR, col = lane % LPR;
  const int nblk = n_req * L;
  const int64_t n_groups = key_off[nblk];
  const int slice = warp % GW;
  // Where the warp's rows of a group lie; the positions of the next group's rows are fetched while this
  // group's rows are on their way.
  struct Place { int64_t row0; int n_rows, r, l, g, pos; };
  auto locate = [&](int64_t gi) {
    Place p{0, 0, 0, 0, 0, 0};
    if (gi >= n_groups) return p;
    int lo = 0, hi = nblk;                           // key_off[lo] <= gi < key_off[hi]
    while (hi - lo > 1) {                            // 32 probes at a time
      const int step = (hi - lo + 31) / 32, at = lo + lane * step;
      const unsigned below = __ballot_sync(kAll, at < hi && key_off[at] <= gi);
      lo += (31 - __clz(below)) * step;
      hi = min(hi, lo + step);
    }
    p.r = lo / L;
    p.l = lo - p.r * L;
    const int len = budget[lo] + Sw;
    const int gpb = (len + GROUP - 1) / GROUP;       // groups per head of this block
    const int rel = (int)(gi - key_off[lo]);
    p.g = rel / gpb;
    const int t0 = (rel - p.g * gpb) * GROUP + slice * 32;
    p.n_rows = max(0, min(32, len - t0));
    p.row0 = row_off[lo] + (int64_t)p.g * len + t0;
    p.pos = p.n_rows > 0 ? pos_packed[p.row0 + min(lane, p.n_rows - 1)] : 0;
    return p;
  };
  const int64_t first = (int64_t)blockIdx.x * (QU_WARPS / GW), stride = (int64_t)gridDim.x * (QU_WARPS / GW);
  Place next = locate(first + warp / GW);
  for (int64_t u0 = first; u0 < n_groups; u0 += stride) {
    const int64_t gi = u0 + warp / GW;
    const Place here = next;
    const int n_rows = here.n_rows, my_pos = here.pos;
    const int64_t row0 = here.row0;
    const size_t head = ((size_t)here.g * T_tokens + reqs[here.r].cu) * D + col * 8;
    const T* kb = reinterpret_cast<const T*>(ptrs.k[here.l]) + head;
    const T* vb = reinterpret_cast<const T*>(ptrs.v[here.l]) + head;
    // rows beyond the last one repeat it (`pos` of the lanes beyond n_rows)
    auto fetch = [&](Oct<T, kVec> (&q)[NB], const T* base, int b) {
#pragma unroll
      for (int j = 0; j < NB; ++j) q[j].load(base + (size_t)(uint32_t)__shfl_sync(kAll, my_pos, (b + j) * RPP + sub) * D);
    };
    // ---- keys: the range of every channel over the group's rows
    float mn[8], mx[8];
    {
      Channels<T> ch;
      ch.clear();
      if (n_rows > 0) {
#pragma unroll 1
        for (int b = 0; b < NIT; b += NB) {
          Oct<T, kVec> q[NB];
          fetch(q, kb, b);
#pragma unroll
          for (int j = 0; j < NB; ++j) ch.add(q[j]);
        }
      }
      ch.get(mn, mx);
    }
    next = locate(gi + stride);
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        mn[e] = fminf(mn[e], __shfl_xor_sync(kAll, mn[e], o));
        mx[e] = fmaxf(mx[e], __shfl_xor_sync(kAll, mx[e], o));
      }
    if constexpr (GW > 1) {
      __syncthreads();                               // the previous round's readers are done
      if (sub == 0)
#pragma unroll
        for (int e = 0; e < 8; ++e) { s_mn[warp][col * 8 + e] = mn[e]; s_mx[warp][col * 8 + e] = mx[e]; }
      __syncthreads();
#pragma unroll
      for (int w = 0; w < GW; ++w)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          mn[e] = fminf(mn[e], s_mn[warp - slice + w][col * 8 + e]);
          mx[e] = fmaxf(mx[e], s_mx[warp - slice + w][col * 8 + e]);
        }
    }
    if (n_rows <= 0) continue;                       // the whole warp; a group's other warps meet it at the barriers above
    {
      f32x2 nz[2][2], rc[2][2], ns[2][2];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const float s0 = scale_of(mn[e], mx[e]), s1 = scale_of(mn[e + 1], mx[e + 1]);
        nz[e / 4][e / 2 % 2] = pack2(-mn[e], -mn[e + 1]);
        rc[e / 4][e / 2 % 2] = pack2(safe_rcp(s0), safe_rcp(s1));
        ns[e / 4][e / 2 % 2] = pack2(-s0, -s1);
        mx[e] = s0;                                  // from here on the scale
        mx[e + 1] = s1;
      }
      if (slice == 0 && sub == 0) {
        float *ks = k_scale + (size_t)gi * D + 8 * col, *kz = k_zero + (size_t)gi * D + 8 * col;
        if constexpr (kVec) {
#pragma unroll
          for (int e = 0; e < 8; e += 4) {
            *reinterpret_cast<float4*>(ks + e) = make_float4(mx[e], mx[e + 1], mx[e + 2], mx[e + 3]);
            *reinterpret_cast<float4*>(kz + e) = make_float4(mn[e], mn[e + 1], mn[e + 2], mn[e + 3]);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) { ks[e] = mx[e]; kz[e] = mn[e]; }
        }
      }
      uint8_t* out = k_codes + (size_t)row0 * (D / 2) + 4 * col;
#pragma unroll 1
      for (int b = 0; b < NIT && b * RPP < n_rows; b += NB) {
        Oct<T, kVec> q[NB];
        fetch(q, kb, b);
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int row = (b + j) * RPP + sub;
          float x[2][4];
          bool odd[2];
          q[j].values(0, x[0]);
          q[j].values(1, x[1]);
          uint32_t c = fast_codes(x[0], nz[0], rc[0], ns[0], odd[0]) | fast_codes(x[1], nz[1], rc[1], ns[1], odd[1]) << 16;
          if (odd[0] || odd[1])
            c = exact_codes(x[0][0], x[0][1], x[0][2], x[0][3], mn[0], mn[1], mn[2], mn[3], mx[0], mx[1], mx[2], mx[3]) |
                exact_codes(x[1][0], x[1][1], x[1][2], x[1][3], mn[4], mn[5], mn[6], mn[7], mx[4], mx[5], mx[6], mx[7]) << 16;
          if (row < n_rows) put_codes<kVec>(out + (size_t)row * (D / 2), c);
        }
      }
    }
    // ---- values: a range per row and group of channels
    constexpr int LG = GROUP / 8;                    // lanes of a group: 4, 8 or 16
    uint8_t* out = v_codes + (size_t)row0 * (D / 2) + 4 * col;
#pragma unroll 1
    for (int b = 0; b < NIT && b * RPP < n_rows; b += NB) {
      Oct<T, kVec> q[NB];
      fetch(q, vb, b);
      MinMax<T> m[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) m[j].set(q[j]);
#pragma unroll
      for (int o = LG / 2; o >= NB; o >>= 1)
#pragma unroll
        for (int j = 0; j < NB; ++j) m[j].merge(m[j].moved(o));
      // afterwards the lane holds the range of pass lane % NB
#pragma unroll
      for (int o = NB / 2; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < o; ++j) {
          const MinMax<T> send = up ? m[j] : m[j + o];
          if (up) m[j] = m[j + o];
          m[j].merge(send.moved(o));
        }
      }
      float zmn, zmx;
      m[0].get(zmn, zmx);
      const float vs = scale_of(zmn, zmx), vr = safe_rcp(vs);
      const int my_row = (b + (lane & (NB - 1))) * RPP + sub;
      if ((lane & (LG - 1)) < NB && my_row < n_rows) {
        const size_t at = (size_t)(row0 + my_row) * (D / GROUP) + col / LG;
        v_scale[at] = vs;
        v_zero[at] = zmn;
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int src = (lane & ~(NB - 1)) + j, row = (b + j) * RPP + sub;
        const float z = __shfl_sync(kAll, zmn, src), rcp = __shfl_sync(kAll, vr, src), s = __shfl_sync(kAll, vs, src);
        const f32x2 nz[2] = {pack2(-z, -z), pack2(-z, -z)}, rc[2] = {pack2(rcp, rcp), pack2(rcp, rcp)},
                    ns[2] = {pack2(-s, -s), pack2(-s, -s)};
        float x[2][4];
        bool odd[2];
        q[j].values(0, x[0]);
        q[j].values(1, x[1]);
        uint32_t c = fast_codes(x[0], nz, rc, ns, odd[0]) | fast_codes(x[1], nz, rc, ns, odd[1]) << 16;
        if (odd[0] || odd[1])
          c = exact_codes(x[0][0], x[0][1], x[0][2], x[0][3], z, z, z, z, s, s, s, s) |
              exact_codes(x[1][0], x[1][1], x[1][2], x[1][3], z, z, z, z, s, s, s, s) << 16;
        if (row < n_rows) put_codes<kVec>(out + (size_t)row * (D / 2), c);
      }
    }
  }
}

template <typename T, int D, bool kVec>
void launch_quant_rows(int grid, cudaStream_t st, int group, const LayerPtrs& ptrs, const int64_t* row_off, const int64_t* key_off,
                       const int32_t* budget, const int32_t* pos, const ReqInfo* reqs, uint8_t* kc, float* ks, float* kz,
                       uint8_t* vc, float* vs, float* vz, int n_req, const cake_config& c, int64_t T_tokens) {
#define CAKE_QUANT(GW)                                                                                                  \
  quant_rows<T, D, GW, kVec><<<grid, QU_WARPS * 32, 0, st>>>(ptrs, row_off, key_off, budget, pos, reqs, kc, ks, kz, vc, vs, vz,  \
                                                             n_req, c.n_layers, c.n_kv_heads, c.window, T_tokens)
  if (group == 32) CAKE_QUANT(1);
  else if (group == 64) CAKE_QUANT(2);
  else if constexpr (D == 128) CAKE_QUANT(4);        // a group is no wider than the head
#undef CAKE_QUANT
}

}  // namespace

int32_t launch_compact_int4(cake_ctx* ctx, int32_t lo, int32_t hi, const LayerPtrs& ptrs, int32_t group,
                            uint8_t* k_codes, float* k_scale, float* k_zero, uint8_t* v_codes,
                            float* v_scale, float* v_zero, int64_t* row_offsets, int64_t* kgroup_offsets,
                            int32_t* positions, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  const int32_t* budget = ctx->d_budget[(ctx->n_evicted - 1) & 1];
  int32_t* pos = positions ? positions : ctx->d_pos_packed;
  int32_t rc = run_offsets(ctx, lo, hi, row_offsets, kgroup_offsets, group, nullptr, st);
  if (rc != CAKE_OK || ctx->n_req == 0 || hi <= lo) return rc;
  rc = run_sorted_positions(ctx, 0, ctx->n_req, lo, hi, row_offsets, pos, 0, st);
  if (rc != CAKE_OK) return rc;
  // vector accesses need rows and key scales on a 16-byte boundary and codes on a 4-byte one
  const bool fp32 = c.dtype == CAKE_DTYPE_FP32;
  uintptr_t in = 0;
  for (int l = lo; l < hi; ++l) in |= (uintptr_t)ptrs.k[l] | (uintptr_t)ptrs.v[l];
  const bool vec = in % 16 == 0 && ((uintptr_t)k_scale | (uintptr_t)k_zero) % 16 == 0 &&
                   ((uintptr_t)k_codes | (uintptr_t)v_codes) % 4 == 0;
  const int grid = ctx->n_sm * (fp32 ? 5 : 6);
#define CAKE_QUANT_ROWS(T, D, V)                                                                                        \
  launch_quant_rows<T, D, V>(grid, st, group, ptrs, row_offsets, kgroup_offsets, budget, pos, ctx->d_req, k_codes, k_scale, \
                             k_zero, v_codes, v_scale, v_zero, ctx->n_req, c, ctx->total_tokens)
  if (fp32 && c.head_dim == 128) { if (vec) CAKE_QUANT_ROWS(float, 128, true); else CAKE_QUANT_ROWS(float, 128, false); }
  else if (fp32) { if (vec) CAKE_QUANT_ROWS(float, 64, true); else CAKE_QUANT_ROWS(float, 64, false); }
  else if (c.head_dim == 128) { if (vec) CAKE_QUANT_ROWS(__nv_bfloat16, 128, true); else CAKE_QUANT_ROWS(__nv_bfloat16, 128, false); }
  else { if (vec) CAKE_QUANT_ROWS(__nv_bfloat16, 64, true); else CAKE_QUANT_ROWS(__nv_bfloat16, 64, false); }
#undef CAKE_QUANT_ROWS
  count_launch();
  return cuda_status(cudaGetLastError());
}

}  // namespace cake
