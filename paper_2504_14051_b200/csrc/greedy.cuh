// Greedy multi-token eviction (Appendix B of the paper, the two-token derivation chained): evict the token whose removal
// changes the current output least, renormalise the weights of the rest, update the output, and score again, k times.
//
// A pick moves the output X = Y / H (Y = sum_j h_j v_j, H = sum_j h_j) by exactly the score of the token it evicts, and by
// the triangle inequality no distance || X - v_j || changes by more than that. So the distances of all tokens are formed
// once (a "build"), and from then on a token's distance is known to within the drift, the sum of the scores evicted since
// it was last formed. A pick forms again only the distances of the tokens that can be the minimum: in the order of their
// lower bounds until the next one is above the smallest score found, usually one. The pick is the same as if all distances had
// been formed again in the picks' own arithmetic (a warp's 32 lanes per row, also where all warps share the work; compared by
// (score bits, position, slot)). The builds' sums, eight lanes per row, only make bounds; the bounds carry margins of 2e-5 for the
// rounding of scores and 5e-7 || X || per pick for that of X.
//
// Likewise only the tokens with small scores at the build can be picked: the `active` ones, found by a radix search, with as
// many of their value rows in shared memory as fit. A pick whose score comes within the drift of the others' smallest score
// is not taken but starts another build; the first pick after a build is always safe.
//
// A thread-block cluster per unit: all CTAs share the two sweeps over the unit's rows (Y, and the distances of a build); the
// picks are one chain of dependent instructions and run on one warp of one CTA, the others wait at the cluster barrier. The
// warp keeps Y and X in registers and w / (1 - w), which all grow together as H falls, from an earlier pick while that has not
// moved a bound by 5e-4. What bounds a pick is the number of its instructions: one warp alone runs straight-line code at about
// four cycles each.
//
// Where bounds do not tell the tokens apart a pick would walk through the list one token after the other; after kAlone of them all
// warps form the other scores at once. 8 units of 4 224 tokens, 128 picks, us (eight warps and 768 active tokens, as it once
// was; one warp; now): log-normal weights 156, 129, 128; equal weights 323, 365, 296; equal weights and 64 different rows
// 783, 5 540, 868; equal rows 4 300, 21 360, 4 270. 900 tokens, 300 of them with weights of 1e-41, 60 picks: 107, 1 303, 221.
// The list holds 256 tokens where it held 768, so long evictions build more often, and are faster all the same: log-normal
// weights, 512 picks 780 -> 553, 2 048 picks 4 270 -> 2 820; equal weights, 1 600 picks 8 540 -> 5 300. What is slower for it is
// long evictions among few different rows of equal weights, where a build lasts only a few picks: 64 rows, 1 600 picks 18.2 -> 23.4 ms.
// 8 units of 4 224 tokens, 128 picks: 709 us with every distance formed at every pick (clusters of 8, rows in shared
// memory, a cluster barrier per pick) -> 149 us on eight warps with two barriers per pick -> 113, of which the sweeps and the
// search are 12. Eight lanes per candidate on one warp, a division per token, upper bounds in a pass of their own: 149 (a pick
// 1 830 cycles: bounds 292, exact score 1 020, though one round per pick); the same without the divisions 137. Earlier
// still: sixteen warps, active tokens in registers, loops unrolled 175; four warps 181; every warp with its own bound and one
// barrier per pick 200 - 211.
#pragma once

#include <cfloat>

#include "common.cuh"
#include "ptx.cuh"

namespace caote {
namespace greedy {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPer = 8;                  // active tokens per lane of the warp that runs the picks
constexpr int kList = 32 * kPer;         // active tokens, at most
constexpr int kWant = kList - 64;        // and what the search asks for, at most
// Scores that the warp of the picks forms alone: 1: 145 us, 2: 135, log-normal weights; 2: 300, 6: 365, equal ones (128 picks, 4 224 tokens).
constexpr int kAlone = 2;
static_assert(kList == 16 * kWarps, "");
constexpr int kMaxTokens = 24576;        // two floats per token in shared memory
constexpr int kMaxC = 8;

inline size_t base_smem_bytes(int cap) { return sizeof(float) * 2 * (((size_t)cap + 3) / 4 * 4) + 16; }

// w / (1 - w) from the un-normalised weight h and the sum H of all.
__device__ __forceinline__ float ratio_of(float h, float H) {
  const float rest = H - h;  // the others' weight (times H)
  const float r = rest > 0.f ? __fdividef(h, rest) : INFINITY;
  return (H > 0.f && h > 0.f) ? r : 0.f;
}
__device__ __forceinline__ float score_of(float h, float dist, float H) {
  const float r = ratio_of(h, H);
  return r == 0.f ? 0.f : r * dist;
}
__device__ __forceinline__ float approx_sqrt(float x) {  // 1 ulp
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A distance (and the drift) as a bound keeps it: finite, also where it overflows or is no number. A token's lower bound is then
// a number: 0, as its score, when its share of the weights underflows to 0, however far it lies.
__device__ __forceinline__ float bound_of(float dist) { return fminf(dist, FLT_MAX); }

// A token in the order of picks: score bits, position, slot; and its number in the list of active tokens.
struct __align__(16) Cand {
  unsigned v, p, s;
  int i;
};
__device__ __forceinline__ bool before(const Cand& a, const Cand& b) {
  return a.v < b.v || (a.v == b.v && (a.p < b.p || (a.p == b.p && a.s < b.s)));
}
// The lane that holds the warp's first token.
__device__ __forceinline__ int first_of(const Cand& c) {
  const unsigned v = __reduce_min_sync(0xffffffffu, c.v);
  unsigned m = __ballot_sync(0xffffffffu, c.v == v);
  if (m & (m - 1u)) {  // a tie, or no token at all
    const unsigned p = __reduce_min_sync(0xffffffffu, c.v == v ? c.p : 0xffffffffu);
    const bool eq = c.v == v && c.p == p;
    const unsigned s = __reduce_min_sync(0xffffffffu, eq ? c.s : 0xffffffffu);
    m = __ballot_sync(0xffffffffu, eq && c.s == s);
  }
  return __ffs((int)m) - 1;
}

// 16 bytes of a row against the same channels of -X (nx: 16-byte aligned), packed fp32 pairs.
template <typename T>
__device__ __forceinline__ float sq_dist16(uint4 raw, const float4* nx) {
  float2 a = make_float2(0.f, 0.f);
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  if constexpr (sizeof(T) == 2) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float4 x = nx[c];
      const float2 d0 = __fadd2_rn(make_float2(__uint_as_float(w[2 * c] << 16), __uint_as_float(w[2 * c] & 0xffff0000u)), make_float2(x.x, x.y));
      const float2 d1 = __fadd2_rn(make_float2(__uint_as_float(w[2 * c + 1] << 16), __uint_as_float(w[2 * c + 1] & 0xffff0000u)), make_float2(x.z, x.w));
      a = __ffma2_rn(d0, d0, a);
      a = __ffma2_rn(d1, d1, a);
    }
  } else {
    const float4 x = nx[0];
    const float2 d0 = __fadd2_rn(make_float2(__uint_as_float(w[0]), __uint_as_float(w[1])), make_float2(x.x, x.y));
    const float2 d1 = __fadd2_rn(make_float2(__uint_as_float(w[2]), __uint_as_float(w[3])), make_float2(x.z, x.w));
    a = __ffma2_rn(d0, d0, a);
    a = __ffma2_rn(d1, d1, a);
  }
  return a.x + a.y;
}

// A lane's channels when a warp shares a row.
template <typename T, int D>
struct __align__(D / 32 * sizeof(T)) LanePiece { T e[D / 32]; };

// The scores of the tokens of `mask` among the warp's 16 of the list, four at a time with eight lanes each, and the first of them:
// to the last bit what a warp per token gives (a lane adds up the parts of four of its lanes in the order of their exchange).
template <typename T, int D>
__device__ __forceinline__ void scores_of(unsigned mask, const T* rows, int rows_smem, const T* Vu, const int* act, const float* th, float* ta,
                                          const unsigned* tp, const float* nX, float H, float drift, Cand* out) {
  constexpr int CPL = D / 32;
  using Piece = LanePiece<T, D>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3, l8 = lane & 7;
  Cand best{0xffffffffu, 0xffffffffu, 0xffffffffu, -1};
#pragma unroll 1
  while (mask) {
    const unsigned m1 = mask & (mask - 1u), m2 = m1 & (m1 - 1u), m3 = m2 & (m2 - 1u);
    const unsigned ms = sub == 0 ? mask : (sub == 1 ? m1 : (sub == 2 ? m2 : m3));
    const int i = 16 * warp + (ms ? __ffs((int)ms) - 1 : 0);  // (a token of the list either way: its first ones are there, or mask is 0)
    const Piece* row = reinterpret_cast<const Piece*>(i < rows_smem ? rows + (size_t)i * D : Vu + (size_t)act[i] * D);
    Piece v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = row[l8 + 8 * c];
    float q[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      q[c] = 0.f;
#pragma unroll
      for (int e = 0; e < CPL; ++e) {
        const float df = to_float(v[c].e[e]) + nX[(l8 + 8 * c) * CPL + e];
        q[c] = fmaf(df, df, q[c]);
      }
    }
    float a = (q[0] + q[2]) + (q[1] + q[3]);
    a += __shfl_xor_sync(0xffffffffu, a, 4);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    if (ms && l8 == 0) {
      const float h = th[i], d = approx_sqrt(a), ro = ratio_of(h, H);
      const Cand c{__float_as_uint(ro == 0.f ? 0.f : ro * d), tp[i], (unsigned)act[i], i};
      if (before(c, best)) best = c;
      if (h > 0.f) ta[i] = bound_of(d + drift);
    }
    mask = m3 & (m3 - 1u);
  }
  if (lane == first_of(best)) out[warp] = best;
}

// This warp's part of sum_j h_j v_j and (at [D]) sum_j h_j over the rows r0 .. r1. (The two sweeps are calls: compiled as a part of the
// kernel their loads were spread out differently with every change of the picks, up to 8 % of a sweep.)
template <typename T, int D>
__device__ __noinline__ void sum_rows(const T* __restrict__ Vu, const float* __restrict__ hu, int r0, int r1, float* part) {
  constexpr int CPL = D / 32;  // channels per lane when a warp shares a row
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float hsum = 0.f, y[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) y[c] = 0.f;
  constexpr int kFly = 8;  // rows in flight per warp
  for (int j0 = r0 + warp; j0 < r1; j0 += kFly * kWarps) {
    float hj[kFly], v[kFly][CPL];
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int j = j0 + u * kWarps;
      hj[u] = (j < r1) ? fmaxf(hu[j], 0.f) : 0.f;
      const T* p = Vu + (size_t)min(j, r1 - 1) * D + lane * CPL;
#pragma unroll
      for (int c = 0; c < CPL; ++c) v[u][c] = to_float(p[c]);
    }
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      hsum += hj[u];
#pragma unroll
      for (int c = 0; c < CPL; ++c) y[c] = fmaf(hj[u], v[u][c], y[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < CPL; ++c) part[lane * CPL + c] = y[c];
  if (lane == 0) part[D] = hsum;  // (every lane added the same weights)
}
// The distances of the rows r0 .. r1 to X, to rank 0's array of them (its address in the cluster: ds0).
template <typename T, int D>
__device__ __noinline__ void distances(const T* __restrict__ Vu, int r0, int r1, const float* nX, uint32_t ds0) {
  constexpr int E = 16 / (int)sizeof(T);  // elements per 16-byte piece
  constexpr int NCH = D / 8 / E;          // pieces per lane when eight lanes share a row: pieces l8, l8 + 8, ...
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3, l8 = lane & 7;
  float4 x[NCH][E / 4];
#pragma unroll
  for (int i = 0; i < NCH; ++i)
#pragma unroll
    for (int e = 0; e < E / 4; ++e) x[i][e] = reinterpret_cast<const float4*>(nX)[(l8 + 8 * i) * (E / 4) + e];
  constexpr int kPasses = 8 / NCH;  // passes of four rows per warp in flight
  for (int j0 = r0 + 4 * warp; j0 < r1; j0 += 4 * kWarps * kPasses) {
    uint4 raw[kPasses][NCH];
#pragma unroll
    for (int u = 0; u < kPasses; ++u) {
      const int j = min(j0 + u * 4 * kWarps + sub, r1 - 1);
#pragma unroll
      for (int i = 0; i < NCH; ++i) raw[u][i] = reinterpret_cast<const uint4*>(Vu + (size_t)j * D)[l8 + 8 * i];
    }
#pragma unroll
    for (int u = 0; u < kPasses; ++u) {
      const int j = j0 + u * 4 * kWarps + sub;
      float a = 0.f;
#pragma unroll
      for (int i = 0; i < NCH; ++i) a += sq_dist16<T>(raw[u][i], x[i]);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      if (l8 == 0 && j < r1) ptx::st_dsmem_f32(ds0 + 4 * j, approx_sqrt(a));
    }
  }
}

// grid = units x C CTAs in clusters of C; rows_smem: value rows that fit behind the two arrays of `cap` floats.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads, 1)
greedy_cluster_kernel(int Hkv, int cap, int rows_smem, const T* __restrict__ V, const float* __restrict__ h_in,
                      const int* __restrict__ len, const int* __restrict__ budget, const int* __restrict__ pos,
                      int* __restrict__ evict_idx, int* __restrict__ order_out, int max_evict, int* __restrict__ n_evict,
                      int* status) {
  constexpr int E = 16 / (int)sizeof(T);  // elements per 16-byte piece
  constexpr int CPL = D / 32;             // channels per lane when a warp shares a row
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ __align__(16) unsigned char gsm[];
  float* hs = reinterpret_cast<float*>(gsm);            // [cap] weight of the token, < 0 once evicted  (rank 0)
  float* ds = hs + (cap + 3) / 4 * 4;                   // [cap] distance at the build                 (rank 0)
  T* rows = reinterpret_cast<T*>(ds + (cap + 3) / 4 * 4);  // [rows_smem][D] value rows of the first active tokens
  __shared__ float Ys[D], part[D + 1], wpart[kWarps][D + 1];
  __shared__ __align__(16) float nX[D];                 // -X
  __shared__ float s_H;
  __shared__ int s_ctl;                                 // after a round of picks: picks done, -1: all
  __shared__ int act[kList];                            // the active tokens: slot,
  __shared__ __align__(16) float th[kList], ta[kList];  // weight (< 0: evicted, or no token), distance + drift when it was formed,
  __shared__ unsigned tp[kList];                        // position
  __shared__ Cand s_cand[kWarps];                       // where all warps form scores: the first of a warp's tokens,
  __shared__ unsigned short s_want[kWarps];             // ... for which of its 16 they are formed, as bits
  __shared__ float s_drift, s_sum;                      // ... at which drift and H
  __shared__ int s_go;                                  // ... 0: the picks have ended
  __shared__ unsigned hist[256];
  __shared__ int s_digit, s_below, s_incl, s_na;
  __shared__ unsigned s_min[kWarps];
  __shared__ int s_cnt[kWarps];

  const int C = (int)ptx::cluster_nctarank(), rank = (int)ptx::cluster_ctarank();
  const int unit = (int)ptx::cluster_id_x(), b = unit / Hkv, hd = unit % Hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = len[b];
  int bud = budget[b];
  if (bud < 1) bud = 1;
  int k = n - bud;
  if (k < 0 || n > cap) k = 0;
  if (k > max_evict) {
    if (tid == 0 && rank == 0) set_status(status, CAOTE_ERR_OVERFLOW);
    k = 0;
  }
  if (hd == 0 && rank == 0 && tid == 0) n_evict[b] = k;
  if (k == 0) return;  // (the whole cluster leaves: no barrier is outstanding)
  const int share = (n + C - 1) / C, r0 = min(n, rank * share), r1 = min(n, r0 + share);  // this CTA's rows in the sweeps
  const T* Vu = V + (size_t)unit * cap * D;
  const float* hu = h_in + (size_t)unit * cap;
  const int* pu = pos ? pos + (size_t)unit * cap : nullptr;

  // ---- H and Y: every CTA its rows, in a fixed order of partial sums ----
  {
    if (rank == 0)
      for (int j = tid; j < n; j += kThreads) hs[j] = fmaxf(hu[j], 0.f);
    sum_rows<T, D>(Vu, hu, r0, r1, wpart[warp]);
    __syncthreads();
    if (tid <= D) {
      float t = 0.f;
      for (int w = 0; w < kWarps; ++w) t += wpart[w][tid];
      part[tid] = t;
    }
  }
  ptx::cluster_sync_all();
  if (rank == 0 && tid <= D) {
    float t = 0.f;
    for (int i = 0; i < C; ++i) t += ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(part + tid), i));
    if (tid < D) Ys[tid] = t; else s_H = t;
  }
  ptx::cluster_sync_all();

  int t = 0;
  while (true) {
    // ================= a build: the distances of all tokens still present to the current output =================
    float H = ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(&s_H), 0));
    {
      const float inv_H = (H > 0.f) ? __fdividef(1.f, H) : 0.f;
      if (tid < D) nX[tid] = -(ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(Ys + tid), 0)) * inv_H);
      __syncthreads();
      distances<T, D>(Vu, r0, r1, nX, ptx::map_to_rank(ptx::smem_u32(ds), 0));
    }
    ptx::cluster_sync_all();

    if (rank == 0) {
      // ---- the active tokens: the smallest (score, position, slot) keys, `want` of them, and at most as many as the list holds ----
      const int present = n - t, rem = k - t, want = min(present, min(rem + 32, kWant));
      unsigned kb = 0u, kp = 0u, ks = 0u;  // the largest key that is taken
      int below = 0;
      for (int pass = 0;; ++pass) {  // eight bits at a time: four passes over the score, four the position, two the slot
        if (tid < 256) hist[tid] = 0u;
        __syncthreads();
        const int at = pass & 3, shift = pass < 8 ? 24 - 8 * at : 8 - 8 * at;
        for (int j = tid; j < n; j += kThreads) {
          const float h = hs[j];
          if (h < 0.f) continue;
          unsigned v = __float_as_uint(score_of(h, ds[j], H)), pre = kb;
          if (pass >= 4) {
            if (v != kb) continue;
            v = (unsigned)(pu ? pu[j] : j);
            pre = kp;
          }
          if (pass >= 8) {
            if (v != kp) continue;
            v = (unsigned)j;
            pre = ks;
          }
          if (shift < 24 && ((v ^ pre) >> (shift + 8)) != 0u) continue;
          atomicAdd(&hist[(v >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (warp == 0) {
          unsigned c[8], sum = 0u;
#pragma unroll
          for (int q = 0; q < 8; ++q) { c[q] = hist[8 * lane + q]; sum += c[q]; }
          unsigned incl = sum;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
          }
          const unsigned need = (unsigned)(want - below);
          const unsigned reach = __ballot_sync(0xffffffffu, need <= incl);
          const int f = reach ? __ffs((int)reach) - 1 : 31;
          if (lane == f) {
            unsigned run = incl - sum;
            int q = 0;
            for (; q < 7 && run + hist[8 * lane + q] < need; ++q) run += hist[8 * lane + q];
            s_digit = 8 * lane + q;
            s_below = below + (int)run;
            s_incl = below + (int)(run + hist[8 * lane + q]);
          }
        }
        __syncthreads();
        const unsigned digit = (unsigned)s_digit << shift;
        if (pass < 4) kb |= digit;
        else if (pass < 8) kp |= digit;
        else ks |= digit;
        below = s_below;
        if (s_incl <= kList || pass == 9) {
          const unsigned ones = (1u << shift) - 1u;
          if (pass < 4) { kb |= ones; kp = 0xffffffffu; ks = 0xffffffffu; }
          else if (pass < 8) { kp |= ones; ks = 0xffffffffu; }
          else ks |= ones;
          break;
        }
      }
      if (tid == 0) s_na = 0;
      __syncthreads();
      float dmin = INFINITY;  // smallest distance among the other tokens
      for (int j0 = 0; j0 < n; j0 += kThreads) {
        const int j = j0 + tid;
        bool in = false;
        if (j < n && hs[j] >= 0.f) {
          const unsigned v = __float_as_uint(score_of(hs[j], ds[j], H));
          in = v < kb;
          if (v == kb) {
            const unsigned p = (unsigned)(pu ? pu[j] : j);
            in = p < kp || (p == kp && (unsigned)j <= ks);
          }
          if (!in) dmin = fminf(dmin, ds[j]);
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&s_na, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (in && at < kList) act[at] = j;  // (the order of the list does not matter: keys decide)
      }
      {
        const unsigned m = __reduce_min_sync(0xffffffffu, __float_as_uint(dmin));
        if (lane == 0) s_min[warp] = m;
      }
      __syncthreads();
      const int na = min(s_na, kList);
      dmin = __uint_as_float(__reduce_min_sync(0xffffffffu, s_min[lane & (kWarps - 1)]));
      const float tau = __uint_as_float(min(kb, 0x7f800000u)), inv_dmin = 1.f / dmin;  // (0 where there are no others)
      for (int i = tid; i < kList; i += kThreads) {
        const int j = i < na ? act[i] : 0;
        th[i] = i < na ? hs[j] : -1.f;
        ta[i] = i < na && hs[j] > 0.f ? bound_of(ds[j]) : INFINITY;  // (no bound: it would be visited after all others)
        tp[i] = (unsigned)(pu ? pu[j] : j);
      }
      for (int idx = tid; idx < min(na, rows_smem) * (D / E); idx += kThreads)
        reinterpret_cast<uint4*>(rows)[idx] = reinterpret_cast<const uint4*>(Vu + (size_t)act[idx / (D / E)] * D)[idx % (D / E)];
      float xn = 0.f;
#pragma unroll
      for (int c = 0; c < CPL; ++c) xn = fmaf(nX[lane * CPL + c], nX[lane * CPL + c], xn);
      xn = sqrtf(warp_sum(xn));
      __syncthreads();

      const bool all_here = na <= rows_smem;
      using Piece = LanePiece<T, D>;
      // ================= picks: one warp =================
      // Lane l looks after the tokens kPer l .. kPer l + 7 of the list and after CPL channels of Y and X, in registers. A pick
      // visits the tokens in the order of their lower bounds, the smallest first, forms the score of each, and ends when the
      // next bound is above the smallest score so far: two rounds, mostly. The number in the list stands in the low bits of a
      // bound, so one reduction over the warp gives both, and the next round's is the smallest key above this one.
      if (warp == 0) {
        float r[kPer], hm = 0.f;  // w / (1 - w) at an earlier H, times 0.99998: a lower bound, since it grows as H falls
        int zeros = 0;            // tokens of weight 0
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          const float h = th[kPer * lane + u];
          r[u] = 1.f;
          hm = fmaxf(hm, h);
          zeros += h == 0.f ? 1 : 0;
        }
        hm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(hm)));
        zeros = __reduce_add_sync(0xffffffffu, zeros);
        float y[CPL], x[CPL];  // Y, -X
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          y[c] = Ys[lane * CPL + c];
          x[c] = nX[lane * CPL + c];
        }
        auto channels = [&](int i, float (&v)[CPL]) {  // this lane's of token i (two loads: the one from shared memory is compiled as such)
          const Piece q = all_here || i < rows_smem ? reinterpret_cast<const Piece*>(rows + (size_t)i * D)[lane]
                                                    : reinterpret_cast<const Piece*>(Vu + (size_t)act[i] * D)[lane];
#pragma unroll
          for (int c = 0; c < CPL; ++c) v[c] = to_float(q.e[c]);
        };
        float drift = 0.f, rest0 = -1.f;  // rest0: H - hm when r was formed, < 0: not yet
        bool fresh = true;
        while (t < k) {
          const float rest = H - hm;  // (what r has grown by since: rest0 / rest, at most)
          if (!(rest0 > 0.f && rest0 < 1.0005f * rest && rest >= 0.05f * H)) {
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
              const float h = th[kPer * lane + u];
              r[u] = h > 0.f ? fminf(0.99998f * ratio_of(h, H), FLT_MAX) : 1.f;
            }
            rest0 = rest;
          }
          int key[kPer];
          {
            const float4 a0 = reinterpret_cast<const float4*>(ta)[2 * lane], a1 = reinterpret_cast<const float4*>(ta)[2 * lane + 1];
            const float av[kPer] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int u = 0; u < kPer; u += 2) {
              const float2 lb = __fmul2_rn(__fadd2_rn(make_float2(av[u], av[u + 1]), make_float2(-drift, -drift)), make_float2(r[u], r[u + 1]));
              key[u] = (__float_as_int(lb.x) & ~(kList - 1)) | (kPer * lane + u);  // (as signed numbers in the order of the bounds;
              key[u + 1] = (__float_as_int(lb.y) & ~(kList - 1)) | (kPer * lane + u + 1);  // below 0 in any order, all of them first)
            }
          }
          int best_v = 0x7fffffff, bi = -1;  // the smallest score so far (its bits) and whose it is
          float he = 0.f, ve[CPL];           // its weight and channels
          auto first = [&](int i, int v) { return bi < 0 || v < best_v || (v == best_v && (tp[i] < tp[bi] || (tp[i] == tp[bi] && act[i] < act[bi]))); };
          auto take = [&](int i, int v) {
            if (first(i, v)) {
              best_v = v;
              bi = i;
              he = th[i];
              channels(i, ve);
            }
          };
          if (zeros > 0) {  // tokens of weight 0 score 0 whatever their distance (they have no bound in the list): the oldest of them
            int mine = -1;
#pragma unroll 1
            for (int i = kPer * lane; i < kPer * lane + kPer; ++i)
              if (th[i] == 0.f && (mine < 0 || tp[i] < tp[mine] || (tp[i] == tp[mine] && act[i] < act[mine]))) mine = i;
            const unsigned p1 = __reduce_min_sync(0xffffffffu, mine >= 0 ? tp[mine] : 0xffffffffu);
            const bool old = mine >= 0 && tp[mine] == p1;
            const unsigned s1 = __reduce_min_sync(0xffffffffu, old ? (unsigned)act[mine] : 0xffffffffu);
            const unsigned m = __ballot_sync(0xffffffffu, old && (unsigned)act[mine] == s1);
            take(__shfl_sync(0xffffffffu, mine, __ffs((int)m) - 1), 0);
          }
          int alone = 0;
          for (unsigned from = 0x80000000u;;) {  // the smallest key not below `from`
            unsigned w = (unsigned)key[0] - from;
#pragma unroll
            for (int u = 1; u < kPer; ++u) w = min(w, (unsigned)key[u] - from);
            const int next = (int)(__reduce_min_sync(0xffffffffu, w) + from);
            if (next < (int)from || (next & ~(kList - 1)) > best_v) break;
            if (__builtin_expect(++alone > kAlone, 0)) {  // bounds that do not tell the tokens apart: all that may still be the one, by all warps
              unsigned mine = 0u;
#pragma unroll
              for (int u = 0; u < kPer; ++u)
                mine |= key[u] >= next && (key[u] & ~(kList - 1)) <= best_v && th[kPer * lane + u] >= 0.f ? 1u << u : 0u;
              const unsigned above = __shfl_down_sync(0xffffffffu, mine, 1);
              if ((lane & 1) == 0) s_want[lane >> 1] = (unsigned short)(mine | (above << kPer));
#pragma unroll
              for (int c = 0; c < CPL; ++c) nX[lane * CPL + c] = x[c];
              if (lane == 0) {
                s_drift = drift;
                s_sum = H;
                s_go = 1;
              }
              asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
              scores_of<T, D>(s_want[0], rows, rows_smem, Vu, act, th, ta, tp, nX, H, drift, s_cand);
              asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
              const Cand c = s_cand[lane & (kWarps - 1)];
              const int l1 = first_of(c), i1 = __shfl_sync(0xffffffffu, c.i, l1), v1 = __shfl_sync(0xffffffffu, (int)c.v, l1);
              if (i1 >= 0) take(i1, v1);
              break;
            }
            const int i = next & (kList - 1);
            const float h = th[i];
            if (h >= 0.f) {
              float v[CPL], q = 0.f;
              channels(i, v);
#pragma unroll
              for (int c = 0; c < CPL; ++c) {
                const float df = v[c] + x[c];
                q = fmaf(df, df, q);
              }
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
              const float d = approx_sqrt(q), ro = ratio_of(h, H);
              const int sv = __float_as_int(ro == 0.f ? 0.f : ro * d);
              if (first(i, sv)) {
                best_v = sv;
                bi = i;
                he = h;
#pragma unroll
                for (int c = 0; c < CPL; ++c) ve[c] = v[c];
              }
              if (lane == 0 && h > 0.f) ta[i] = bound_of(d + drift);
            }
            if (next == 0x7fffffff) break;
            from = (unsigned)next + 1u;
          }
          if (bi < 0) {         // no active token is left
            if (fresh) t = k;   // (cannot happen with k < n)
            break;
          }
          const float sc = __int_as_float(best_v);
          if (!fresh && !(sc <= tau * (1.f - drift * inv_dmin) * 0.99999f)) break;  // another token may be smaller: build again
          // ---- evict: Y -= h_e v_e, H -= h_e ----
          H -= he;
          const float inv_H = (H > 0.f) ? __fdividef(1.f, H) : 0.f;
#pragma unroll
          for (int c = 0; c < CPL; ++c) {
            y[c] -= he * ve[c];
            x[c] = -(y[c] * inv_H);
          }
          zeros -= he == 0.f ? 1 : 0;
          __syncwarp();  // (th has been read)
          if (lane == 0) {
            const int e = act[bi];
            ta[bi] = INFINITY;
            th[bi] = -1.f;
            hs[e] = -1.f;
            if (order_out) order_out[(size_t)unit * max_evict + t] = e;
          }
          __syncwarp();
          drift += sc * 1.0001f + 5e-7f * (xn + drift);
          fresh = false;
          ++t;
        }
#pragma unroll
        for (int c = 0; c < CPL; ++c) Ys[lane * CPL + c] = y[c];
        if (lane == 0) s_go = 0;
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
      } else {
        while (true) {  // (the warp that runs the picks ends it: the same barriers in the same order on both sides)
          asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
          if (s_go == 0) break;
          scores_of<T, D>(s_want[warp], rows, rows_smem, Vu, act, th, ta, tp, nX, s_sum, s_drift, s_cand);
          asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
        }
      }
      __syncthreads();
      if (tid == 0) {
        s_H = H;
        s_ctl = t < k ? t : -1;
      }
    }
    ptx::cluster_sync_all();
    t = ptx::ld_dsmem_s32(ptx::map_to_rank(ptx::smem_u32(&s_ctl), 0));
    if (t < 0) break;
  }
  ptx::cluster_sync_all();  // (nobody reads rank 0's shared memory any more)
  if (rank != 0) return;
  // ---- the evicted slots in ascending order (the layout caote_compact expects) ----
  int* out = evict_idx + (size_t)unit * max_evict;
  int run = 0;
  for (int j0 = 0; j0 < n; j0 += kThreads) {
    const int j = j0 + tid;
    const bool gone = j < n && hs[j] < 0.f;
    const unsigned m = __ballot_sync(0xffffffffu, gone);
    if (lane == 0) s_cnt[warp] = __popc(m);
    __syncthreads();
    int before = run;
    for (int w = 0; w < kWarps; ++w) {
      if (w < warp) before += s_cnt[w];
      run += s_cnt[w];
    }
    if (gone) out[before + __popc(m & ((1u << lane) - 1u))] = j;
    __syncthreads();
  }
}

}  // namespace greedy
}  // namespace caote
