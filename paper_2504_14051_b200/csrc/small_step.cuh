// The whole decode step (append, scoring, selection of at most one token, FILL compaction, length update) in one launch for
// the single-query shapes that the tensor-core cluster kernel has no form for: fp32, groups of more than 8 heads, or of 8
// with carried scores; short units. fp32 CUDA-core arithmetic as on the any-shape path (generic_score.cuh, whose routines it
// uses), but the passes of a unit meet in a thread-block cluster instead of in global memory: a CTA takes a run of the
// unit's tiles of 64 tokens, keeps their logits in shared memory from the attention pass to the scores, and leaves its
// (maximum, sum, partial output) where the others read it through distributed shared memory. What
// bounds it is latency: 2 units of 255 fp32 tokens, head_dim 64, take 14.0 us here, and 21.1 in the five launches of the
// any-shape path (31 with the host, which is the longer side there).
#pragma once

#include "common.cuh"
#include "generic_score.cuh"
#include "ptx.cuh"

namespace caote {
namespace small {

using generic::kKT;
using generic::kRT;
constexpr int kThreads = 256;
constexpr int kMaxC = 8;
constexpr int kMaxTiles = 4;  // tiles of one CTA

inline int cluster_size(int tiles) {
  int c = 1;
  while (c < kMaxC && c < tiles) c *= 2;
  return c;
}

template <typename T>
struct Args {
  const T *q, *k_new, *v_new;
  T *K, *V;
  float* base;
  int *pos, *len, *n_seen;  // pos, n_seen, vsum may be null
  const int* budget;
  float *o, *scores;
  int *evict_idx, *n_evict, *ticket;
  float* vsum;
};

inline size_t smem_bytes(int D, int tiles) {
  const int LD = D + 4;
  return sizeof(float) * ((size_t)kRT * LD + 2 * kKT * LD + (size_t)tiles * kRT * kKT + kRT * kKT + kRT * D + D + 8 + 2 * kRT +
                          kKT + kThreads + 2 * kMaxC * kRT + kMaxC * kRT + 4 * kRT + D + 4) + 16 * (kThreads / 32) * kMaxC + 64;
}

// grid = units x C CTAs in clusters of C; tiles: most tiles of a CTA.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
small_step_kernel(Dims dm, Args<T> sa, int tiles, int* status) {
  constexpr int LD = D + 4, OC = D / 16, YP = kThreads / D, E = 16 / (int)sizeof(T), kChunks = D / E;
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;                   // [kRT][LD]
  float* Ks = Qs + kRT * LD;          // [kKT][LD], later the merged outputs [G][D]
  float* Vs = Ks + kKT * LD;          // [kKT][LD]
  float* Ls = Vs + kKT * LD;          // [tiles][kRT][kKT] logits
  float* Ps = Ls + tiles * kRT * kKT; // [kRT][kKT]
  float* po = Ps + kRT * kKT;         // [kRT][D] this CTA's partial outputs        (read by the peers)
  float* py = po + kRT * D;           // [D + 8] its share of sum_j base_j v_j, at [D] of sum_j base_j   (read by the peers)
  float* pml = py + D + 8;            // [kRT][2] its (max logit, sum of the others)  (read by the peers)
  float* bs = pml + 2 * kRT;          // [kKT]
  float* red = bs + kKT;              // [kThreads]
  float* ml = red + kThreads;         // [C][kRT][2]
  float* fac = ml + 2 * kMaxC * kRT;  // [C][kRT] weight of a CTA's partial output
  float* st = fac + kMaxC * kRT;      // [kRT][4] max, 1 / sum, share of all but the top key
  float* Xs = st + 4 * kRT;           // [D + 4]; at [D] the sum of the carried scores
  uint4* cand = reinterpret_cast<uint4*>(Xs + D + 4);  // [C][warps] (rank 0)

  const int C = (int)ptx::cluster_nctarank(), rank = (int)ptx::cluster_ctarank();
  const int unit = (int)ptx::cluster_id_x(), b = unit / dm.Hkv, h = unit % dm.Hkv, G = dm.G;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, r = tid >> 4, c0 = tid & 15;
  const int mode = dm.base_mode;
  const bool carried = mode == CAOTE_BASE_ACCUM || mode == CAOTE_BASE_EXTERNAL;
  T* Ku = sa.K + (size_t)unit * dm.cap * D;
  T* Vu = sa.V + (size_t)unit * dm.cap * D;
  float* bu = sa.base ? sa.base + (size_t)unit * dm.cap : nullptr;
  int* pu = sa.pos ? sa.pos + (size_t)unit * dm.cap : nullptr;

  // ---- append: the CTA that has the last tile ----
  uint4 row = make_uint4(0u, 0u, 0u, 0u);
  if (tid < 2 * kChunks) row = reinterpret_cast<const uint4*>((tid < kChunks ? sa.k_new : sa.v_new) + (size_t)unit * D)[tid % kChunks];
  for (int idx = tid; idx < kRT * (D / 4); idx += kThreads) {
    const int rr = idx / (D / 4), c4 = idx % (D / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rr < G) v = load4(sa.q + ((size_t)b * dm.Hq + h * G + rr) * D + c4 * 4);
    *reinterpret_cast<float4*>(Qs + rr * LD + c4 * 4) = v;
  }
  const int n0 = __ldcg(sa.len + b);
  const bool fits = n0 >= 0 && n0 < dm.cap;
  const int n = n0 + (fits ? 1 : 0);
  const bool ok = n > 0 && n <= dm.cap;
  if (tid == 0 && rank == 0) {
    if (!fits) set_status(status, CAOTE_ERR_OVERFLOW);
    if (!ok && n != 0) set_status(status, CAOTE_ERR_BAD_LENGTH);
    if (unit == 0) status[kStatTagIndex] = kStatNone;
  }
  const int nt = ok ? (n + kKT - 1) / kKT : 0, per = (nt + C - 1) / C;
  const int t0 = min(nt, rank * per), t1 = min(nt, t0 + per);
  if (fits && t0 < t1 && t1 == nt) {
    if (tid < 2 * kChunks) reinterpret_cast<uint4*>((tid < kChunks ? Ku : Vu) + (size_t)n0 * D)[tid % kChunks] = row;
    if (tid == 128 && bu) bu[n0] = 0.f;
    if (tid == 129 && pu) pu[n0] = sa.n_seen ? __ldcg(sa.n_seen + b) : n0;
  }

  // ---- attention over this CTA's tiles (as in generic::attn_partial_kernel) ----
  float m_run = -INFINITY, l_rest = 0.f, o_acc[OC], y_acc = 0.f, hb_acc = 0.f;
#pragma unroll
  for (int i = 0; i < OC; ++i) o_acc[i] = 0.f;
  for (int t = t0; t < t1; ++t) {
    const int kt = t * kKT;
    __syncthreads();
    generic::stage_rows<T, D, LD>(Ks, Ku + (size_t)kt * D, kKT, n - kt);
    generic::stage_rows<T, D, LD>(Vs, Vu + (size_t)kt * D, kKT, n - kt);
    if (carried && tid < kKT) bs[tid] = (kt + tid < n) ? bu[kt + tid] : 0.f;
    __syncthreads();
    float s1[1][4], mx = -INFINITY;
    generic::logits<D, LD, 1>(Qs + r * LD, Ks + c0 * LD, dm.scale, s1);
    float(&s)[4] = s1[0];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (r >= G || kt + c0 + 16 * i >= n) s[i] = -INFINITY;
      Ls[((t - t0) * kRT + r) * kKT + c0 + 16 * i] = s[i];
      mx = fmaxf(mx, s[i]);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float m_new = fmaxf(m_run, mx);
    const bool new_top = mx > m_run;
    const float corr = (m_run == -INFINITY) ? 0.f : expf(m_run - m_new);
    float lsum = 0.f;
    bool found = false;  // the first key of the tile at the new maximum is left out of the sum
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float p = (s[i] == -INFINITY) ? 0.f : expf(s[i] - m_new);
      Ps[r * kKT + c0 + 16 * i] = p;
      const unsigned at_top = (__ballot_sync(0xffffffffu, new_top && s[i] == m_new) >> (tid & 16)) & 0xffffu;
      const bool skip = !found && at_top != 0u && (int)(__ffs(at_top) - 1) == c0;
      found |= at_top != 0u;
      lsum += skip ? 0.f : p;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    l_rest = l_rest * corr + ((new_top && m_run != -INFINITY) ? corr : 0.f) + lsum;
    m_run = m_new;
#pragma unroll
    for (int i = 0; i < OC; ++i) o_acc[i] *= corr;
    __syncthreads();
    if (r < G) {
      for (int j = 0; j < kKT; ++j) {
        const float p = Ps[r * kKT + j];
#pragma unroll
        for (int x = 0; x < OC / 4; ++x) {
          const float4 v = *reinterpret_cast<const float4*>(Vs + j * LD + 64 * x + c0 * 4);
          o_acc[4 * x] = fmaf(p, v.x, o_acc[4 * x]);
          o_acc[4 * x + 1] = fmaf(p, v.y, o_acc[4 * x + 1]);
          o_acc[4 * x + 2] = fmaf(p, v.z, o_acc[4 * x + 2]);
          o_acc[4 * x + 3] = fmaf(p, v.w, o_acc[4 * x + 3]);
        }
      }
    }
    if (carried) {
      for (int j = tid / D; j < kKT; j += YP) y_acc = fmaf(bs[j], Vs[j * LD + tid % D], y_acc);
      if (tid < kKT) hb_acc += bs[tid];
    }
  }
  if (c0 == 0) {
    pml[2 * r] = m_run;
    pml[2 * r + 1] = l_rest;
  }
#pragma unroll
  for (int x = 0; x < OC / 4; ++x)
    *reinterpret_cast<float4*>(po + r * D + 64 * x + c0 * 4) = make_float4(o_acc[4 * x], o_acc[4 * x + 1], o_acc[4 * x + 2], o_acc[4 * x + 3]);
  if (carried) {
    __syncthreads();  // bs is read by every thread until here
    red[tid] = y_acc;
    if (tid < kKT) bs[tid] = hb_acc;
    __syncthreads();
    if (tid < D) {
      float y = 0.f;
      for (int p = 0; p < YP; ++p) y += red[p * D + tid];
      py[tid] = y;
    }
    if (warp == kThreads / 32 - 1) {
      const float hb = warp_sum(bs[lane] + bs[lane + 32]);
      if (lane == 0) py[D] = hb;
    }
  }
  ptx::cluster_sync_all();

  // ---- merge: every CTA for itself; the rows of o are dealt to the CTAs ----
  if (tid < 2 * kRT * C) ml[tid] = ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(pml + tid % (2 * kRT)), tid / (2 * kRT)));
  __syncthreads();
  if (tid < kRT) {
    float mx = -INFINITY, rest = 0.f;
    for (int i = 0; i < C; ++i) mx = fmaxf(mx, ml[(i * kRT + tid) * 2]);
    bool top_seen = false;  // the first CTA at the overall maximum keeps its top key apart; the others' join the rest
    for (int i = 0; i < C; ++i) {
      const float m = ml[(i * kRT + tid) * 2], f = (m == -INFINITY) ? 0.f : expf(m - mx);
      rest = fmaf(ml[(i * kRT + tid) * 2 + 1], f, rest);
      if (m == mx && !top_seen) top_seen = true;
      else rest += f;
      fac[i * kRT + tid] = f;
    }
    const float inv_l = 1.f / (rest + 1.f);
    for (int i = 0; i < C; ++i) fac[i * kRT + tid] *= inv_l;
    st[4 * tid] = mx;
    st[4 * tid + 1] = inv_l;
    st[4 * tid + 2] = rest * inv_l;
  }
  __syncthreads();
  float* Os = Ks;
  for (int idx = tid; idx < G * (D / 4); idx += kThreads) {
    const int rr = idx / (D / 4), c = 4 * (idx % (D / 4));
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kMaxC; ++i) {
      if (i < C) {
        const float4 v = ptx::ld_dsmem_v4(ptx::map_to_rank(ptx::smem_u32(po + rr * D + c), i));
        const float f = fac[i * kRT + rr];
        a.x = fmaf(v.x, f, a.x); a.y = fmaf(v.y, f, a.y); a.z = fmaf(v.z, f, a.z); a.w = fmaf(v.w, f, a.w);
      }
    }
    *reinterpret_cast<float4*>(Os + rr * D + c) = a;
    if (ok && rr % C == rank) *reinterpret_cast<float4*>(sa.o + ((size_t)b * dm.Hq + h * G + rr) * D + c) = a;
  }
  __syncthreads();
  if (tid <= D) {
    const int rows = mode == CAOTE_BASE_EXTERNAL ? 0 : G;
    float x = 0.f, hb = 0.f;
    if (tid < D)
      for (int rr = 0; rr < rows; ++rr) x += Os[rr * D + tid];
    if (carried)
      for (int i = 0; i < C; ++i) {
        x += ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(py + tid), i));
        hb += ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(py + D), i));
      }
    const float H = (float)rows + hb;
    float res = H > 0.f ? x / H : 0.f;
    if (sa.vsum && tid < D)  // FastCAOTE: the mean of the cached values (the running sum does not hold the new row yet)
      res = (sa.vsum[(size_t)unit * D + tid] + (fits ? to_float(sa.v_new[(size_t)unit * D + tid]) : 0.f)) / (float)max(n, 1);
    Xs[tid] = tid < D ? res : hb;
  }
  __syncthreads();

  // ---- scores of this CTA's tokens (four threads per token), the tile that is still in shared memory first ----
  unsigned best_v = 0u, best_p = 0u;
  int best_s = -1;
  {
    const float hb = Xs[D], Htot = (mode == CAOTE_BASE_EXTERNAL ? 0.f : (float)G) + hb;
    const int key = tid >> 2, part = tid & 3;
    for (int t = t1 - 1; t >= t0; --t) {
      const int j = t * kKT + key;
      if (t != t1 - 1) {
        __syncthreads();
        generic::stage_rows<T, D, LD>(Vs, Vu + (size_t)t * kKT * D, kKT, n - t * kKT);
        __syncthreads();
      }
      float hj = 0.f, rest = 0.f, d2 = 0.f;
      if (j < n) {
        if (mode != CAOTE_BASE_EXTERNAL)
          for (int rr = part; rr < G; rr += 4) {
            const float sl = Ls[((t - t0) * kRT + rr) * kKT + key];
            const float a = expf(sl - st[4 * rr]) * st[4 * rr + 1];
            hj += a;
            rest += (sl == st[4 * rr]) ? st[4 * rr + 2] : 1.f - a;
          }
#pragma unroll
        for (int c = 0; c < D / 4; c += 4) {  // this thread's channels: part * 4 + 16 i
          const float4 v = *reinterpret_cast<const float4*>(Vs + key * LD + 4 * c + 4 * part);
          const float4 x = *reinterpret_cast<const float4*>(Xs + 4 * c + 4 * part);
          const float d0 = x.x - v.x, d1 = x.y - v.y, dd = x.z - v.z, d3 = x.w - v.w;
          d2 = fmaf(d0, d0, fmaf(d1, d1, fmaf(dd, dd, fmaf(d3, d3, d2))));
        }
      }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        hj += __shfl_xor_sync(0xffffffffu, hj, o);
        rest += __shfl_xor_sync(0xffffffffu, rest, o);
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      }
      if (part == 0 && j < n) {
        if (carried) {
          const float bj = bu[j];
          rest += hb - bj;
          hj += bj;
          if (mode == CAOTE_BASE_ACCUM) bu[j] = hj;
        }
        float ratio = 0.f;
        if (Htot > 0.f && hj > 0.f) ratio = (rest > 0.f) ? hj / rest : INFINITY;
        const float sc = (ratio == 0.f) ? 0.f : ((ratio == INFINITY) ? INFINITY : ratio * sqrtf(d2));
        sa.scores[(size_t)unit * dm.cap + j] = sc;
        first_candidate(best_v, best_p, best_s, __float_as_uint(sc), (unsigned)(pu ? __ldcg(pu + j) : j), j);
      }
    }
  }
  // ---- the warp's candidate to rank 0, which selects and compacts ----
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    first_candidate(best_v, best_p, best_s, __shfl_xor_sync(0xffffffffu, best_v, o), __shfl_xor_sync(0xffffffffu, best_p, o),
                    __shfl_xor_sync(0xffffffffu, best_s, o));
  if (lane == 0) ptx::st_dsmem_v4(ptx::map_to_rank(ptx::smem_u32(cand + rank * (kThreads / 32) + warp), 0), make_uint4(best_v, best_p, (uint32_t)best_s, 0u));
  ptx::cluster_sync_all();
  if (rank != 0) return;
  int bud = __ldg(sa.budget + b);
  if (bud < 1) bud = 1;
  int k = ok ? max(n - bud, 0) : 0;
  if (k > 1) {  // (launched for calls that take one eviction at most)
    if (tid == 0) set_status(status, CAOTE_ERR_OVERFLOW);
    k = 0;
  }
  if (tid == 0 && h == 0) sa.n_evict[b] = k;
  int s = -1;
  if (k == 1) {
    unsigned v = 0u, p = 0u;
    for (int i = lane; i < C * (kThreads / 32); i += 32) first_candidate(v, p, s, cand[i].x, cand[i].y, (int)cand[i].z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      first_candidate(v, p, s, __shfl_xor_sync(0xffffffffu, v, o), __shfl_xor_sync(0xffffffffu, p, o), __shfl_xor_sync(0xffffffffu, s, o));
  }
  if (sa.vsum) {  // the new row joins the running sum, the evicted one leaves it
    if (tid < D) {
      float x = sa.vsum[(size_t)unit * D + tid];
      if (fits) x += to_float(sa.v_new[(size_t)unit * D + tid]);
      if (s >= 0) x -= to_float(Vu[(size_t)s * D + tid]);
      sa.vsum[(size_t)unit * D + tid] = x;
    }
    __syncthreads();
  }
  if (s >= 0) {
    if (tid == 0) sa.evict_idx[unit] = s;
    const int last = n - 1;
    if (s != last) {
      if (warp == 1 && lane < kChunks) reinterpret_cast<uint4*>(Ku + (size_t)s * D)[lane] = __ldcg(reinterpret_cast<const uint4*>(Ku + (size_t)last * D) + lane);
      if (warp == 2 && lane < kChunks) reinterpret_cast<uint4*>(Vu + (size_t)s * D)[lane] = __ldcg(reinterpret_cast<const uint4*>(Vu + (size_t)last * D) + lane);
      if (warp == 3 && lane == 0 && bu) bu[s] = __ldcg(bu + last);
      if (warp == 3 && lane == 1 && pu) pu[s] = __ldcg(pu + last);
    }
  }
  // the cluster that finishes last (a ticket, which it also resets) moves the lengths on
  __shared__ int s_last;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(sa.ticket, 1) == dm.units - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int i = tid; i < dm.B; i += kThreads) {
      const int l0 = __ldcg(sa.len + i), more = (l0 >= 0 && l0 < dm.cap) ? 1 : 0;
      sa.len[i] = l0 + more - __ldcg(sa.n_evict + i);
      if (sa.n_seen) sa.n_seen[i] += more;
    }
    if (tid == 0) *sa.ticket = 0;
  }
}

}  // namespace small
}  // namespace caote
