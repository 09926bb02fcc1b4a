// What follows a layer's scores: its preference, the budgets of its stage (device side), and its pooled
// indicators with their distribution, from which the per-head top-k of the eviction is found where a retained
// set is read.
#include "cake_internal.cuh"

#include <math_constants.h>

#include <algorithm>
#include <cstddef>
#include <cstring>

namespace cake {
namespace {

__device__ inline void raise_status(int32_t* status, int32_t code) { atomicCAS(status, 0, code); }

__device__ inline double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// --------------------------------------------------------------- pool + bins
// When a layer arrives, its pooled indicators are histogrammed: "the top b" are then all values of the buckets
// before the one that contains the b-th, and the best part of that bucket.

// Token ranges of the pooling items: a request's tokens in at most `want` equal runs, a
// multiple of kChunkKeys long.
__device__ inline int split_span(int N, int want) {
  const int chunks = (N + kChunkKeys - 1) / kChunkKeys;
  const int ns = min(chunks, want);
  return ns > 0 ? (chunks + ns - 1) / ns * kChunkKeys : kChunkKeys;
}

// The CTAs of arrive_layer take a whole SM each, 1024 threads in four teams that work on items of their own.
// (As CTAs of a team each they spread over all the SMs that are free in the moment between two score
// launches, and the next one, whose CTAs need whole SMs, waits for them: 136 against 119 us per 128K layer.
// As one team of 1024 an SM has a single chain of scans and barriers at a time: with 256 lists of 2K tokens 97 us
// beside the scoring, 43 as it is; 36 by themselves.)
constexpr int TEAMS = 4;
constexpr int TEAM_THREADS = 256;
constexpr int TEAM_WARPS = TEAM_THREADS / 32;
__device__ __forceinline__ void team_sync() {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / TEAM_THREADS)), "n"(TEAM_THREADS) : "memory");
}
// Exclusive scan of one int per thread of the team; *total gets the sum.
__device__ inline int team_excl_scan(int v, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x % TEAM_THREADS) >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) warp_tot[warp] = inc;
  team_sync();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < TEAM_WARPS; ++w) {
    const int t = warp_tot[w];
    before += w < warp ? t : 0;
    all += t;
  }
  *total = all;
  team_sync();
  return before + inc - v;
}

constexpr int PH_PER = 4;                            // consecutive tokens per thread and pass
constexpr int kTileTok = 4096;                       // tokens of a run on their way to shared memory at a time

struct AllocArgs {           // budgets of one stage
  const double* dP;          // [req][L]
  const int32_t* prev;       // budgets of the stage before
  int32_t* cur;
  int32_t* status;
  int64_t seats;             // B' = B_total - L * S_w
  double slope;
  int L, alloc_mode;
};

struct FinalizeArgs {        // preference of the layer from the score kernels' partial sums
  const float* colpart;      // (sum p log2 p, sum var) of every part of the column pass
  const int32_t* pair_seg;   // tensor-core path: [pairs + 1] first pass-B segment; null on the SIMT path,
                             //   whose parts are the request's score units
  const float* hrow;         // [pair][128] sum_j p log2 p of every window row (tile order), or null: the
                             //   entropy then comes from the column pass (supplied denominators, SIMT)
  double* headsum;           // [req][H_q][2] scratch
  double* dH; double* dV; double* dP;
  int32_t* status;
  int on;                    // 0: indicators were supplied, there is nothing to finalise
  int budgets;               // compute the stage's budgets as well
  int parts;                 // CTAs that share a request's heads (divides H_q)
  uint32_t* arrivals;        // [req] counters of a request's finished parts (zero at rest)
  int rows, Hq;
  double inv_tau1, inv_tau2;
};

constexpr int kMaxCand = 1024;
struct AllocSmem {
  double P[CAKE_MAX_LAYERS];
  int64_t lo[CAKE_MAX_LAYERS];
  int32_t off[CAKE_MAX_LAYERS + 1];
  int32_t win[CAKE_MAX_LAYERS];
  double c_val[kMaxCand];
  int32_t c_lay[kMaxCand];
  double red[2][TEAM_WARPS];
  int last, n_cand;
  int64_t need;
};
template <int NT, typename Sync>
__device__ void allocate_request(const AllocArgs& A, const ReqInfo& rq, int req, int stage, const double* p_stage, AllocSmem& S,
                                 Sync sync);

// H_h = -ln2 * sum p*log2(p), V_h = sum_j Var_i of the query heads h_lo .. h_hi - 1 of a request, a warp
// or several per head; the CTA that completes a request's last heads takes the means over the heads and
// P = H^(1/tau1) * V^(1/tau2) (Eq. 4-6), then the budgets of the stage that this layer completes.  All
// sums run in a fixed order in double precision.
__device__ void finalize_heads(const FinalizeArgs& F, const AllocArgs& A, const ReqInfo& rq, int req, int part, int layer,
                               int Hkv, AllocSmem& S) {
  constexpr int W = TEAM_WARPS;
  const int tid = threadIdx.x % TEAM_THREADS, lane = tid & 31, warp = tid >> 5;
  const int G = F.Hq / Hkv, n_h = F.Hq / F.parts, h_lo = part * n_h;
  // the other layers' preferences, for the budgets: on their way while the sums are formed
  if (F.budgets)
    for (int l = tid; l < layer; l += TEAM_THREADS) S.P[l] = __ldcg(&A.dP[(size_t)req * A.L + l]);
  int wph = 1;                                       // warps per head
  while (wph * 2 * n_h <= W) wph *= 2;
  double* hs = F.headsum + (size_t)req * F.Hq * 2;
  for (int h0 = 0; h0 < n_h; h0 += W / wph) {
    const int h = h_lo + h0 + warp / wph, sub = warp % wph;
    double a = 0.0, b = 0.0;
    if (h < h_lo + n_h) {
      const int g = h / G, hl = h - g * G, pair = req * Hkv + g;
      const float2* part_at = reinterpret_cast<const float2*>(F.colpart);
      int count, stride;
      if (F.pair_seg) {
        const int s_lo = F.pair_seg[pair];
        part_at += (size_t)s_lo * kScoreWarps * G + hl;
        count = (F.pair_seg[pair + 1] - s_lo) * kScoreWarps;
        stride = G;
      } else {
        part_at += ((size_t)rq.unit0 * Hkv + g) * G + hl;
        count = rq.nunits;
        stride = Hkv * G;
      }
      for (int i0 = sub * 32; i0 < count; i0 += 32 * 8 * wph) {      // eight loads per lane in flight
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = i0 + u * 32 * wph + lane;
          v[u] = i < count ? __ldcg(part_at + (size_t)i * stride) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) { a += (double)v[u].x; b += (double)v[u].y; }
      }
      if (F.hrow) {
        a = 0.0;
        if (sub == 0)
          for (int r = hl + lane * G; r < F.rows; r += 32 * G) a += (double)__ldcg(&F.hrow[(size_t)pair * 128 + r]);
      }
      a = warp_sum_f64(a);
      b = warp_sum_f64(b);
    }
    if (wph > 1) {
      if (lane == 0) { S.red[0][warp] = a; S.red[1][warp] = b; }
      team_sync();
      if (sub == 0 && lane == 0)
        for (int w = 1; w < wph; ++w) { a += S.red[0][warp + w]; b += S.red[1][warp + w]; }
      team_sync();
    }
    if (h < h_lo + n_h && sub == 0 && lane == 0) { hs[2 * h] = -0.6931471805599453 * a; hs[2 * h + 1] = b; }
  }
  __threadfence();
  team_sync();
  if (F.parts > 1) {
    if (tid == 0) {
      S.last = atomicAdd(&F.arrivals[req], 1u) + 1u == (uint32_t)F.parts ? 1 : 0;
      if (S.last) F.arrivals[req] = 0;
    }
    team_sync();
    if (!S.last) return;
    __threadfence();
  }
  double P = 0.0;
  if (warp == 0) {
    double H = 0.0, V = 0.0;
    for (int h = lane; h < F.Hq; h += 32) { H += __ldcg(&hs[2 * h]); V += __ldcg(&hs[2 * h + 1]); }
    H = warp_sum_f64(H) / (double)F.Hq;
    V = warp_sum_f64(V) / (double)F.Hq;
    P = (F.inv_tau1 == 1.0 ? H : pow(H, F.inv_tau1)) * (F.inv_tau2 == 1.0 ? V : pow(V, F.inv_tau2));
    if (lane == 0) {
      F.dH[(size_t)req * A.L + layer] = H;
      F.dV[(size_t)req * A.L + layer] = V;
      F.dP[(size_t)req * A.L + layer] = P;
      if (!(P >= 0.0) || isinf(P)) raise_status(F.status, CAKE_ERR_NONFINITE);
    }
  }
  if (F.budgets) allocate_request<TEAM_THREADS>(A, rq, req, layer, &P, S, [] { team_sync(); });
}

// What happens to a layer between its scores and its eviction, in one launch of a grid that fits the
// SMs the next layer's score kernel leaves free (a grid beyond those would sit on SMs that kernel
// needs whole, and hold up all of its CTAs); its CTAs take items in turn:
//   - the preference and the stage's budgets of a request (first, their chain of steps is the longest);
//   - a run of a request's tokens of one KV head: store[g][t] = pool(raw[g][.]) over the request's
//     non-window tokens, +inf on the window (Section 4.3); with do_pool = 0 the pooled values are
//     already there.  A thread owns PH_PER consecutive tokens per pass.  The bucket histogram of
//     the (request, head) is accumulated in `hist`; the CTA that adds the last run turns it into
//     bucket offsets, `prefix`.
// Nothing here depends on the budgets, and nothing else is done for an eviction: which tokens a budget keeps is
// found where a retained set is read (sorted_positions).  Placing every layer's values in bucket order was a launch
// of its own per layer, 6 to 60 us on the few SMs that the score kernel leaves free.
// R = pool_kernel / 2 when that is at most 3, else -1 (any kernel size, one global read per tap).
struct ArriveArgs {
  const float* raw;
  float* store;
  uint16_t* codes;
  const ReqInfo* reqs;
  uint32_t* hist;
  uint32_t* arrivals;
  int32_t* prefix;
  int n_req, want, layer, L, Hkv, kp, mode, do_pool;
  int64_t T, code_T;
};
struct alignas(16) ArriveSmem {   // of a team
  union { uint32_t sh[kBins]; AllocSmem alloc; };
  float tile[2][kTileTok + 8];   // tokens jb - 4 .. jb + kTileTok + 3 of the tile at jb
  int warp_tot[TEAM_WARPS];
  int last;
};
template <int R>
__global__ void __launch_bounds__(TEAMS * TEAM_THREADS)
arrive_layer(const ArriveArgs Q, const FinalizeArgs F, const AllocArgs B) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int team = (int)threadIdx.x / TEAM_THREADS, tid = threadIdx.x % TEAM_THREADS;
  ArriveSmem& S = reinterpret_cast<ArriveSmem*>(smem_raw)[team];
  uint32_t* sh = S.sh;
  const int n_fin = F.on ? Q.n_req * F.parts : 0, n_items = n_fin + Q.n_req * Q.Hkv * Q.want;
  const int layer = Q.layer, L = Q.L, Hkv = Q.Hkv, kp = Q.kp, mode = Q.mode, do_pool = Q.do_pool;
  const int64_t T = Q.T;
  const float* raw = Q.raw;
  for (int item = team * gridDim.x + blockIdx.x; item < n_items; item += TEAMS * gridDim.x) {
    team_sync();                                   // the item before is done with shared memory
    if (item < n_fin) {
      const int r = item / F.parts;
      finalize_heads(F, B, Q.reqs[r], r, item - r * F.parts, layer, Hkv, S.alloc);
      continue;
    }
    const int split = (item - n_fin) % Q.want, pair = (item - n_fin) / Q.want;
    const int req = pair / Hkv, g = pair - req * Hkv;
    const ReqInfo rq = Q.reqs[req];
    const int span = split_span(rq.N, Q.want), nsplit = (rq.N + span - 1) / span;
    if (split >= nsplit) continue;
    for (int b = tid; b < kBins; b += TEAM_THREADS) sh[b] = 0;
    team_sync();
    const float* src = raw + (size_t)g * T + rq.cu;
    float* dst = Q.store + (size_t)g * T + rq.cu;
    uint16_t* code = Q.codes + (size_t)g * Q.code_T + code_row(rq.cu, req);
    const int t0 = split * span, t1 = min(rq.N, t0 + span);
    // Writes four tokens and counts their buckets.  Neighbours often share a bucket, so a run is counted
    // once, at its first token; without branches (with them a warp issued some 300 instructions for its
    // 128 tokens, and the pooling was bound by that).
    const bool vec = (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
    auto put = [&](int j0, const float (&out)[PH_PER]) {
      if (j0 + PH_PER <= rq.n && j0 + PH_PER <= t1) {
        if (do_pool) {
          if (vec) {
            *reinterpret_cast<float4*>(dst + j0) = make_float4(out[0], out[1], out[2], out[3]);
          } else {
#pragma unroll
            for (int e = 0; e < PH_PER; ++e) dst[j0 + e] = out[e];
          }
        }
        uint32_t key[PH_PER];
        int q[PH_PER];
#pragma unroll
        for (int e = 0; e < PH_PER; ++e) {
          key[e] = ordered_key(out[e]);
          q[e] = bucket_of(key[e]);
        }
        *reinterpret_cast<uint2*>(code + j0) = make_uint2(__byte_perm(key[0], key[1], 0x7632), __byte_perm(key[2], key[3], 0x7632));
        const bool s1 = q[1] != q[0], s2 = q[2] != q[1], s3 = q[3] != q[2];
        atomicAdd(&sh[q[0]], s1 ? 1u : s2 ? 2u : s3 ? 3u : 4u);
        if (s1) atomicAdd(&sh[q[1]], s2 ? 1u : s3 ? 2u : 3u);
        if (s2) atomicAdd(&sh[q[2]], s3 ? 1u : 2u);
        if (s3) atomicAdd(&sh[q[3]], 1u);
      } else {
#pragma unroll
        for (int e = 0; e < PH_PER; ++e) {
          const int j = j0 + e;
          if (j < t1 && j >= rq.n) {
            dst[j] = CUDART_INF_F;
          } else if (j < t1) {
            const uint32_t key = ordered_key(out[e]);
            if (do_pool) dst[j] = out[e];
            code[j] = (uint16_t)(key >> 16);
            atomicAdd(&sh[bucket_of(key)], 1u);
          }
        }
      }
    };
    if constexpr (R >= 0) {
      // A run comes in tiles, the next one on its way while one is pooled (a thread that fetched its own
      // tokens with their neighbours waited for every four of them: 28 us for 8K tokens beside a score
      // kernel that keeps the memory system busy).
      const float* in = do_pool ? src : dst;
      const float pad = mode == CAKE_POOL_MAX ? -CUDART_INF_F : 0.f;
      auto fetch = [&](int buf, int jb) {
        const int cnt = min(kTileTok, t1 - jb) + 8;
        for (int i = tid; i < cnt; i += TEAM_THREADS) {
          const int j = jb - 4 + i;
          if (j >= 0 && j < rq.n) copy_async4(&S.tile[buf][i], in + j);
          else S.tile[buf][i] = pad;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
      fetch(0, t0);
      for (int jb = t0, buf = 0; jb < t1; jb += kTileTok, buf ^= 1) {
        if (jb + kTileTok < t1) {
          fetch(buf ^ 1, jb + kTileTok);
          asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        team_sync();
        for (int q = tid; q < kTileTok / PH_PER && jb + q * PH_PER < t1; q += TEAM_THREADS) {
          float v[12];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const float4 f = reinterpret_cast<const float4*>(S.tile[buf])[q + i];
            v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
          }
          float out[PH_PER];
#pragma unroll
          for (int e = 0; e < PH_PER; ++e) {
            float m = v[4 + e];
            if (do_pool) {
              m = v[4 + e - R];
#pragma unroll
              for (int x = 1; x <= 2 * R; ++x) m = mode == CAKE_POOL_MAX ? fmaxf(m, v[4 + e - R + x]) : m + v[4 + e - R + x];
              if (mode != CAKE_POOL_MAX) m /= (float)kp;
            }
            out[e] = m;
          }
          put(jb + q * PH_PER, out);
        }
        team_sync();
      }
    } else {
      const int r = kp >> 1;
      for (int j0 = t0 + tid * PH_PER; j0 < t1; j0 += TEAM_THREADS * PH_PER) {
        float out[PH_PER];
#pragma unroll 1
        for (int e = 0; e < PH_PER; ++e) {
          const int j = j0 + e;
          float m = 0.f;
          if (j < rq.n) {
            if (do_pool) {
              const int a = max(0, j - r), b = min(rq.n, j + r + 1);
              m = src[a];
              for (int x = a + 1; x < b; ++x) m = mode == CAKE_POOL_MAX ? fmaxf(m, src[x]) : m + src[x];
              if (mode != CAKE_POOL_MAX) m /= (float)kp;
            } else {
              m = dst[j];
            }
          }
          out[e] = m;
        }
        put(j0, out);
      }
    }
    team_sync();
    uint32_t* gh = Q.hist + (size_t)pair * kBins;
    if (nsplit > 1) {
      for (int b = tid; b < kBins; b += TEAM_THREADS)
        if (sh[b]) atomicAdd(&gh[b], sh[b]);
      __threadfence();
      team_sync();
      if (tid == 0) {
        const uint32_t old = atomicAdd(&Q.arrivals[pair], 1u);
        S.last = (old + 1u == (uint32_t)nsplit) ? 1 : 0;
      }
      team_sync();
      if (!S.last) continue;
      __threadfence();
    }
    // bucket offsets: prefix[i] = values in buckets before i
    int32_t* pf = Q.prefix + (((size_t)req * L + layer) * Hkv + g) * (kBins + 1);
    // (a warp takes a run of the buckets, 32 at a time, so that all accesses are consecutive)
    constexpr int PER = kBins / TEAM_THREADS;
    const int lane = tid & 31, first = (tid >> 5) * (32 * PER) + lane;
    int cnt[PER], sum = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      cnt[e] = (int)(nsplit > 1 ? __ldcg(&gh[first + 32 * e]) : sh[first + 32 * e]);
      sum += cnt[e];
    }
    int total;
    int run = team_excl_scan(sum, S.warp_tot, &total);
    run = __shfl_sync(0xffffffffu, run, 0);            // elements before the warp's run
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      int inc = cnt[e];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
      }
      pf[first + 32 * e] = run + inc - cnt[e];
      run += __shfl_sync(0xffffffffu, inc, 31);
      if (nsplit > 1) gh[first + 32 * e] = 0;          // ready for the next layer
    }
    if (tid == 0) pf[kBins] = total;
    if (nsplit > 1 && tid == 0) Q.arrivals[pair] = 0;
  }
}

// ----------------------------------------------------------------- allocate
// Number of s in [0, lim) with P/(s + 1/2) >= x (IEEE double division).  The estimate is nearly always right, and
// the two divisions that confirm it do not wait for one another.
__device__ inline int64_t count_ge(double P, double x, int64_t lim) {
  if (!(P > 0.0) || isinf(x)) return 0;
  const double est = floor(P / x - 0.5) + 1.0;
  int64_t c = est < 0.0 ? 0 : (est > (double)lim ? lim : (int64_t)est);
  const double last = P / ((double)(c - 1) + 0.5), next = P / ((double)c + 0.5);
  if ((c == 0 || last >= x) && (c == lim || next < x)) return c;
  while (c > 0 && P / ((double)(c - 1) + 0.5) < x) --c;
  while (c < lim && P / ((double)c + 0.5) >= x) ++c;
  return c;
}

__device__ inline int64_t warp_sum64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Budgets of one request, by NT threads: the first warp's, and all of them where candidates are ranked.  Webster /
// Sainte-Lague: the `seats` largest priorities
// P_l/(s+1/2) win, ties to the lower layer then the lower s.  The common divisor
// is bracketed analytically (sum_l round(P_l/x) is within L/2 of sum(P)/x), the few
// priorities inside the bracket are ranked exactly; if the bracket ever fails the
// threshold is found by bisection over the bit patterns of the doubles.  p_stage: preference of the
// newest layer where this launch has just computed it (the others are in S.P then), else null (all of them are
// in dP).
//
// Bound: latency, a chain of double divisions, sums over the warp and the ranking.  With a bracket of L on either
// side, ranked by one warp with two comparisons a candidate, and the preferences fetched here it took 8.5 us at 32
// layers, the longest step behind a layer's scores.
template <int NT, typename Sync>
__device__ void allocate_request(const AllocArgs& A, const ReqInfo& rq, int req, int stage, const double* p_stage, AllocSmem& S,
                                 Sync sync) {
  const int tid = (int)threadIdx.x % NT, lane = tid & 31, L = A.L;
  const int64_t seats = A.seats;
  int32_t* status = A.status;
  double* sP = S.P;
  int64_t* s_lo = S.lo;
  int32_t *s_off = S.off, *s_win = S.win;
  double* c_val = S.c_val;
  int32_t* c_lay = S.c_lay;
  const int La = stage + 1;
  int32_t* out = A.cur + (size_t)req * L;
  const int32_t* old = A.prev + (size_t)req * L;
  // what one warp does before the ranking: the candidates, or (0) the budgets themselves
  auto prepare = [&]() -> int {
    for (int l = La + lane; l < L; l += 32) out[l] = 0;
    bool bad = false;
    bool anypos = false;
    double SP = 0.0;
    for (int l = lane; l < La; l += 32) {
      // what the split is proportional to: the preference (Eq. 7 / Eq. 9), or one of the fixed
      // patterns of the paper's allocation ablation (Section 5.3)
      double p = !p_stage ? A.dP[(size_t)req * L + l] : l == stage ? *p_stage : sP[l];
      if (A.alloc_mode == CAKE_ALLOC_UNIFORM) p = 1.0;
      else if (A.alloc_mode == CAKE_ALLOC_PYRAMID) p = L > 1 ? 1.0 + A.slope * (double)(L - 1 - 2 * l) / (double)(L - 1) : 1.0;
      sP[l] = p;
      if (!(p >= 0.0) || isinf(p)) bad = true;
      if (p > 0.0) anypos = true;
      SP += p;
    }
    bad = __any_sync(0xffffffffu, bad);
    anypos = __any_sync(0xffffffffu, anypos);
    __syncwarp();
    if (bad) {                                   // keep the previous stage's budgets
      raise_status(status, CAKE_ERR_NONFINITE);
      for (int l = lane; l < La; l += 32) out[l] = (l < stage && stage > 0) ? old[l] : 0;
      return 0;
    }
    if (rq.keep_all) {
      for (int l = lane; l < La; l += 32) out[l] = rq.n;
      return 0;
    }
    if (!anypos) {
      SP = 0.0;
      for (int l = lane; l < La; l += 32) { sP[l] = 1.0; SP += 1.0; }
      __syncwarp();
    }
    if (seats <= 0) {
      for (int l = lane; l < La; l += 32) out[l] = 0;
      return 0;
    }
    SP = warp_sum_f64(SP);
    if (isinf(SP)) {
      raise_status(status, CAKE_ERR_NONFINITE);
      for (int l = lane; l < La; l += 32) out[l] = (l < stage && stage > 0) ? old[l] : 0;
      return 0;
    }
    const int64_t lim = seats + La + 8;
    const int64_t margin = (La + 1) / 2 + 1;     // half a seat per layer, and one for the roundings
    const double x_lo = SP / (double)(seats + margin);
    const double x_hi = seats > margin ? SP / (double)(seats - margin) : CUDART_INF;
    int64_t clo = 0, chi = 0;
    for (int l = lane; l < La; l += 32) {
      const int64_t a = count_ge(sP[l], x_hi, lim);
      const int64_t b = count_ge(sP[l], x_lo, lim);
      s_lo[l] = a;
      s_win[l] = 0;
      const int64_t nc = b - a;
      s_off[l + 1] = (int32_t)(nc > kMaxCand ? kMaxCand + 1 : nc);
      clo += a;
      chi += b;
    }
    clo = warp_sum64(clo);
    chi = warp_sum64(chi);
    __syncwarp();
    const bool bracket_ok = clo <= seats && chi >= seats && (chi - clo) <= kMaxCand;
    if (bracket_ok) {
      // offsets of the layers' candidates: inclusive scan, 32 layers at a time
      int carry = 0;
      for (int l0 = 0; l0 < La; l0 += 32) {
        int v = l0 + lane < La ? s_off[l0 + lane + 1] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += t;
        }
        if (l0 + lane < La) s_off[l0 + lane + 1] = carry + v;
        carry += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) s_off[0] = 0;
      __syncwarp();
      for (int l = lane; l < La; l += 32) {
        const int base = s_off[l], cnt = s_off[l + 1] - base;
        for (int e = 0; e < cnt; ++e) {
          const int64_t s = s_lo[l] + e;
          c_val[base + e] = sP[l] / ((double)s + 0.5);
          c_lay[base + e] = l;
        }
      }
      if (lane == 0) S.need = seats - clo;
      return s_off[La] > 0 ? s_off[La] : -1;     // -1: nothing to rank, but the counts to write
    }
    // Fallback: T = largest double x with C(x) >= seats, by bisection on bit patterns.
    double pmax = 0.0;
    for (int l = 0; l < La; ++l) pmax = fmax(pmax, sP[l]);
    unsigned long long lo_bits = 1ull;                                   // C(lo) >= seats
    unsigned long long hi_bits = (unsigned long long)__double_as_longlong(pmax / 0.5) + 1ull;  // C(hi) = 0
    if (hi_bits > 0x7FF0000000000000ull) hi_bits = 0x7FF0000000000000ull;
    for (int it = 0; it < 70 && hi_bits - lo_bits > 1ull; ++it) {
      const unsigned long long mid = lo_bits + ((hi_bits - lo_bits) >> 1);
      const double x = __longlong_as_double((long long)mid);
      int64_t c = 0;
      for (int l = lane; l < La; l += 32) c += count_ge(sP[l], x, lim);
      c = warp_sum64(c);
      if (c >= seats) lo_bits = mid; else hi_bits = mid;
    }
    const double Tthr = __longlong_as_double((long long)lo_bits);
    const double Tnext = __longlong_as_double((long long)(lo_bits + 1ull));
    int64_t gt_sum = 0;
    for (int l = lane; l < La; l += 32) {
      const int64_t gt = count_ge(sP[l], Tnext, lim);
      const int64_t ge = count_ge(sP[l], Tthr, lim);
      s_lo[l] = gt;
      s_win[l] = (int32_t)(ge - gt);            // 0 or 1: priorities strictly decrease in s
      gt_sum += gt;
    }
    gt_sum = warp_sum64(gt_sum);
    __syncwarp();
    if (lane == 0) {
      int64_t need = seats - gt_sum;
      for (int l = 0; l < La; ++l) {
        int64_t b = s_lo[l];
        if (s_win[l] > 0 && need > 0) { b += 1; need -= 1; }
        out[l] = (int32_t)(b < (int64_t)rq.n ? b : (int64_t)rq.n);
      }
    }
    return 0;
  };
  if (tid < 32) {
    const int n = prepare();
    if (lane == 0) S.n_cand = n;
  }
  sync();
  const int ncand = S.n_cand;
  if (ncand == 0) return;
  const int64_t need = S.need;
  // candidates stand in the order of the tie rule (layer, then s): equal ones are ahead if they stand before
  for (int c = tid; c < ncand; c += NT) {
    const double v = c_val[c];
    int ahead = 0;
#pragma unroll 8
    for (int o = 0; o < c; ++o) ahead += c_val[o] >= v ? 1 : 0;
#pragma unroll 8
    for (int o = c + 1; o < ncand; ++o) ahead += c_val[o] > v ? 1 : 0;
    if (ahead < need) atomicAdd(&s_win[c_lay[c]], 1);
  }
  sync();
  for (int l = tid; l < La; l += NT) {
    const int64_t b = s_lo[l] + s_win[l];
    out[l] = (int32_t)(b < (int64_t)rq.n ? b : (int64_t)rq.n);
  }
}

__global__ void allocate_budgets(const AllocArgs A, const ReqInfo* __restrict__ reqs, int stage) {
  __shared__ AllocSmem S;
  allocate_request<32>(A, reqs[blockIdx.x], blockIdx.x, stage, nullptr, S, [] { __syncwarp(); });
}

static_assert(offsetof(ArriveSmem, tile) % 16 == 0 && sizeof(ArriveSmem) % 16 == 0, "tiles are read 16 bytes at a time");

}  // namespace

// CTAs of arrive_layer, and runs per (request, head).  While the next layer is scored they run on the
// SMs its kernel leaves free; behind the last layer the whole device is theirs.
static void cascade_shape(const cake_ctx* ctx, int32_t layer, int extra_items, int* want, int* grid) {
  const int pairs = ctx->n_req * ctx->cfg.n_kv_heads;
  int slots = ctx->n_sm;
  if (layer + 1 < ctx->cfg.n_layers) slots = ctx->use_tc ? std::max(8, ctx->n_sm - ctx->n_tc_ctas) : ctx->n_sm / 4;
  int w = std::max(1, slots * TEAMS / std::max(1, pairs));
  w = std::min(w, (ctx->max_n_tokens + kChunkKeys - 1) / kChunkKeys);
  *want = std::max(1, w);
  *grid = std::min(slots, pairs * *want + extra_items);
}

static AllocArgs alloc_args(const cake_ctx* ctx, int32_t stage) {
  const cake_config& c = ctx->cfg;
  AllocArgs A;
  A.dP = ctx->d_P;
  A.prev = ctx->d_budget[(stage + 1) & 1];
  A.cur = ctx->d_budget[stage & 1];
  A.status = ctx->d_status;
  A.seats = ctx->sel_budget;
  A.slope = (double)c.pyramid_slope;
  A.L = c.n_layers;
  A.alloc_mode = c.alloc_mode;
  return A;
}

// Pooling + bucket histogram of layer `layer`; with `finalize` also the layer's preference, with
// `budgets` the budgets of its stage too.
int32_t launch_arrive(cake_ctx* ctx, int32_t layer, bool do_pool, bool finalize, bool budgets, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  if (ctx->n_req == 0) return CAKE_OK;
  FinalizeArgs F;
  memset(&F, 0, sizeof(F));
  F.Hq = c.n_q_heads;
  if (finalize) {
    F.on = 1;
    F.budgets = budgets ? 1 : 0;
    F.colpart = ctx->d_colpart[layer % ctx->score_depth];
    F.pair_seg = ctx->use_tc ? ctx->d_tc_index + (ctx->n_req * c.n_kv_heads + 1) : nullptr;
    F.hrow = ctx->use_tc && ctx->hhead_from_rows ? ctx->d_hrow[layer % ctx->score_depth] : nullptr;
    F.headsum = ctx->d_headsum;
    F.arrivals = ctx->d_arrivals + ctx->max_pairs;
    // the chain of loads and sums is the longest item of the launch: one team per request took 14 us of 16 at 8K tokens
    // and 22 of 24 at 32K, the pooling beside it 7 and 13
    F.parts = ctx->n_fin_parts;
    F.dH = ctx->d_H; F.dV = ctx->d_V; F.dP = ctx->d_P;
    F.status = ctx->d_status;
    F.rows = ctx->rows;
    F.inv_tau1 = 1.0 / (double)c.tau1;
    F.inv_tau2 = 1.0 / (double)c.tau2;
  }
  ArriveArgs Q;
  Q.raw = ctx->d_raw[layer % ctx->score_depth];
  Q.store = layer_store(ctx, layer);
  Q.codes = layer_codes(ctx, layer);
  Q.reqs = ctx->d_req;
  Q.hist = ctx->d_hist;
  Q.arrivals = ctx->d_arrivals;
  Q.prefix = ctx->d_prefix;
  Q.n_req = ctx->n_req; Q.layer = layer; Q.L = c.n_layers; Q.Hkv = c.n_kv_heads;
  Q.kp = c.pool_kernel; Q.mode = c.pool_mode; Q.do_pool = do_pool ? 1 : 0;
  Q.T = ctx->total_tokens;
  Q.code_T = code_tokens(ctx->total_tokens, ctx->n_req);
  int grid;
  cascade_shape(ctx, layer, finalize ? ctx->n_req * F.parts : 0, &Q.want, &grid);
  const AllocArgs B = alloc_args(ctx, layer);
  static PerDeviceOnce attr;
  if (attr.need(ctx->device)) {
    const int bytes = (int)(TEAMS * sizeof(ArriveSmem));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(arrive_layer<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(arrive_layer<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(arrive_layer<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(arrive_layer<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    CAKE_CUDA_TRY(cudaFuncSetAttribute(arrive_layer<-1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    attr.mark(ctx->device);
  }
  switch (c.pool_kernel / 2) {
    case 0: arrive_layer<0><<<grid, TEAMS * TEAM_THREADS, TEAMS * sizeof(ArriveSmem), st>>>(Q, F, B); break;
    case 1: arrive_layer<1><<<grid, TEAMS * TEAM_THREADS, TEAMS * sizeof(ArriveSmem), st>>>(Q, F, B); break;
    case 2: arrive_layer<2><<<grid, TEAMS * TEAM_THREADS, TEAMS * sizeof(ArriveSmem), st>>>(Q, F, B); break;
    case 3: arrive_layer<3><<<grid, TEAMS * TEAM_THREADS, TEAMS * sizeof(ArriveSmem), st>>>(Q, F, B); break;
    default: arrive_layer<-1><<<grid, TEAMS * TEAM_THREADS, TEAMS * sizeof(ArriveSmem), st>>>(Q, F, B); break;
  }
  count_launch();
  return cuda_status(cudaGetLastError());
}

int32_t launch_allocate(cake_ctx* ctx, int32_t stage, cudaStream_t st) {
  if (ctx->n_req == 0) return CAKE_OK;
  allocate_budgets<<<ctx->n_req, 32, 0, st>>>(alloc_args(ctx, stage), ctx->d_req, stage);
  count_launch();
  return cuda_status(cudaGetLastError());
}

}  // namespace cake
