// Generic scoring path: any I/O dtype (bf16 / fp32), head_dim 64 or 128, any block size m, any group
// size up to 16. Plain fp32 CUDA-core arithmetic, three launches:
//
//   attn_partial  split-KV flash attention over tiles of 16 or 64 query rows x 64 keys: per (unit, split,
//                 row) running max, running sum and un-normalised partial output; row tile 0 also
//                 accumulates sum_j base_j v_j and sum_j base_j for the base modes that carry scores.
//   attn_combine  merges the splits: final (max, 1/sum) per row, attention output o, and per 32-row
//                 chunk the sum of the output rows that define the base score.
//   score_pass    key-major: a CTA owns 64 cached tokens, recomputes their logits against every
//                 counted query row with the same dot-product routine, sums alpha over rows into h_j,
//                 applies the base mode, and writes c_j = w_j/(1-w_j) * ||X - v_j|| once.
//
// X = sum_j w_j v_j is never formed by a pass of its own: because w is a non-negative combination of
// attention rows (plus the carried base score), X = (sum of the counted output rows + sum_j base_j v_j)
// / (number of counted rows + sum_j base_j).
//
// All reductions run in a fixed order, so results are bit-reproducible from run to run.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace caote {
namespace generic {

constexpr int kRT = 16;          // query rows per tile
constexpr int kKT = 64;          // keys per tile
constexpr int kThreads = 256;
constexpr int kCombineThreads = 512;

struct Scratch {
  float* part_ml;  // [units][splits][Rpad][2]   (max logit, sum of exp(s - max) over all keys but the first one at the max)
  float* part_o;   // [units][splits][Rpad][D]
  float* part_y;   // [units][splits][D]
  float* part_hb;  // [units][splits]
  float* stats;    // [units][Rpad][4]   (max, 1/sum, (sum without the row's top key) / sum, unused)
  float* osum;     // [units][chunks][D]
  float* ytot;     // [units][D]
  float* hbtot;    // [units]
  int splits, Rpad, chunks, chunk_rows;  // chunk_rows: rows of a combine CTA
};

inline int round_up(int x, int a) { return (x + a - 1) / a * a; }

// Query rows per thread (x 16 = rows of a tile). What bounds the tiles is what shared memory delivers to registers; a thread
// with four rows uses every K and V value four times. fp32 steps, head_dim 128, 2 048 tokens, us with one row and with four:
// 16 units of 896 rows 2001, 969; 4 units of 896 rows 991, 355; 32 units of 64 rows 344, 218; 8 units of 45 rows 134, 116;
// but 8 units of 32 rows 92, 98: half of the tile is empty and there are fewer tiles for the SMs.
constexpr int kManyRows = 4;
inline int rows_per_thread(int rows) { return rows >= 40 ? kManyRows : 1; }

// Number of key splits: enough CTAs (tiles of `rows` query rows) to fill the machine a few times over, never more splits than
// there are spans of `span` keys in the cache.
inline int choose_splits(const Dims& dm, int rows, int span) {
  const int row_tiles = (dm.R + rows - 1) / rows;
  const long ctas = (long)dm.units * row_tiles;
  int s = (int)(((long)g_sm_count * 4 + ctas - 1) / ctas);
  const int max_by_cap = (dm.cap + span - 1) / span;
  if (s > max_by_cap) s = max_by_cap;
  if (s > 32) s = 32;
  if (s < 1) s = 1;
  return s;
}

inline size_t carve_as(const Dims& dm, char* base, Scratch* out, int splits, int chunk_rows) {
  Scratch s;
  s.splits = splits;
  s.chunk_rows = chunk_rows;
  s.Rpad = round_up(dm.R, kRT);
  s.chunks = (dm.R + chunk_rows - 1) / chunk_rows;
  size_t off = 0;
  auto take = [&](size_t n_floats) {
    float* p = reinterpret_cast<float*>(base + off);
    off = align_up(off + n_floats * sizeof(float), 256);
    return p;
  };
  const size_t us = (size_t)dm.units * s.splits;
  s.part_ml = take(us * s.Rpad * 2);
  s.part_o = take(us * s.Rpad * dm.D);
  s.part_y = take(us * dm.D);
  s.part_hb = take(us);
  s.stats = take((size_t)dm.units * s.Rpad * 4);
  s.osum = take((size_t)dm.units * s.chunks * dm.D);
  s.ytot = take((size_t)dm.units * dm.D);
  s.hbtot = take((size_t)dm.units);
  if (out) *out = s;
  return off;
}

// Splits down to single tiles (a tile is a chain of its own latency: 256 tokens, 2 units: 9 us in spans of two, 5 in one) and
// chunks of 16 rows, as far as the scratch allows. Every split keeps a full set of partial outputs, and a thread of four rows
// asks for up to four times as many splits, so the scratch is bounded by what tiles of 16 rows, spans of two tiles and
// chunks of 32 rows take; for fp32, whose main path this is, by the built-in array of caote_score_static where that is more.
// (bf16 gets here with sums of errors over blocks of queries and with the few forms that the tensor-core kernels leave;
// without the bound a cache of 8 units, 512 rows and 4 224 slots held 21.5 MB for it instead of 8.5.)
inline size_t carve(const Dims& dm, bool f32, char* base, Scratch* out) {
  size_t bound = carve_as(dm, nullptr, nullptr, choose_splits(dm, kRT, 2 * kKT), 32);
  if (f32 && bound < CAOTE_STATIC_SCRATCH_BYTES - kHeaderBytes) bound = CAOTE_STATIC_SCRATCH_BYTES - kHeaderBytes;
  for (int splits = choose_splits(dm, kRT * rows_per_thread(dm.R), kKT); splits > 1; --splits)
    if (carve_as(dm, nullptr, nullptr, splits, 16) <= bound) return carve_as(dm, base, out, splits, 16);
  return carve_as(dm, base, out, 1, carve_as(dm, nullptr, nullptr, 1, 16) <= bound ? 16 : 32);
}

// scale * <q, k> over D channels, in one fixed order, from fp32 rows in shared memory, for RPT queries and four keys 16 rows
// apart (a row is fetched once for all of them). All passes call this, so a logit has the same bits in all of them.
template <int D, int LD, int RPT>
__device__ __forceinline__ void logits(const float* __restrict__ qrow, const float* __restrict__ krow, float scale, float (&s)[RPT][4]) {
#pragma unroll
  for (int u = 0; u < RPT; ++u) s[u][0] = s[u][1] = s[u][2] = s[u][3] = 0.f;
#pragma unroll(RPT == 1 ? 8 : 4)
  for (int c = 0; c < D; c += 4) {
    float4 a[RPT];
#pragma unroll
    for (int u = 0; u < RPT; ++u) a[u] = *reinterpret_cast<const float4*>(qrow + u * 16 * LD + c);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 b = *reinterpret_cast<const float4*>(krow + i * 16 * LD + c);
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        s[u][i] = fmaf(a[u].x, b.x, s[u][i]);
        s[u][i] = fmaf(a[u].y, b.y, s[u][i]);
        s[u][i] = fmaf(a[u].z, b.z, s[u][i]);
        s[u][i] = fmaf(a[u].w, b.w, s[u][i]);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < RPT; ++u)
#pragma unroll
    for (int i = 0; i < 4; ++i) s[u][i] *= scale;
}

// Stage `rows` rows of D elements (global, dtype T) into shared memory as fp32 with row stride LD;
// rows at or beyond `valid_rows` are zero-filled.
template <typename T, int D, int LD>
__device__ __forceinline__ void stage_rows(float* dst, const T* src, int rows, int valid_rows) {
  constexpr int V4 = D / 4;
  for (int idx = threadIdx.x; idx < rows * V4; idx += blockDim.x) {
    const int r = idx / V4, c4 = idx % V4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < valid_rows) v = load4(src + (size_t)r * D + c4 * 4);
    *reinterpret_cast<float4*>(dst + r * LD + c4 * 4) = v;
  }
}

// Row r of a unit: query head g = r / m, query i = r % m.
__device__ __forceinline__ size_t q_offset(const Dims& dm, int b, int h, int r) {
  const int g = r / dm.m, i = r % dm.m;
  return (((size_t)b * dm.Hq + h * dm.G + g) * dm.m + i) * dm.D;
}

// Floats per key of the table of numerators (many rows: a thread's rows side by side, 16-byte columns on different banks).
__host__ __device__ constexpr int p_pitch(int rpt) { return rpt == 1 ? kRT : kRT * rpt + 4; }

// Thread (r = tid / 16, c0 = tid % 16) has rows r + 16 u of the tile, keys c0 + 16 i, channels 4 c0 + 64 x.
template <typename T, int D, int RPT>
__global__ void __launch_bounds__(kThreads, RPT == 1 ? 0 : 2)
attn_partial_kernel(Dims dm, const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                    const int* __restrict__ len, const float* __restrict__ base, Scratch sc, int* status) {
  constexpr int LD = D + 4;
  constexpr int OC = D / 16;  // output channels per thread (two float4 for D = 128, one for D = 64)
  constexpr int kR = kRT * RPT, kPitch = p_pitch(RPT);
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;
  float* Ks = Qs + kR * LD;
  float* Vs = RPT == 1 ? Ks + kKT * LD : Ks;  // (many rows: V takes the place of K, so that two CTAs fit an SM)
  float* Ps = Vs + kKT * LD;                  // one row per thread: [row][key]; many: [key][kPitch], r * RPT + u in it
  float* bs = Ps + kKT * kPitch;              // kKT base values
  float* red = bs + kKT;        // kThreads floats

  const int unit = blockIdx.z, split = blockIdx.y, rt = blockIdx.x;
  const int b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b];
  if (threadIdx.x == 0 && unit == 0 && split == 0 && rt == 0) status[kStatTagIndex] = kStatNone;
  if (n == 0) return;
  if (n < dm.m || n > dm.cap) {
    if (threadIdx.x == 0) set_status(status, CAOTE_ERR_BAD_LENGTH);
    return;
  }
  const bool use_base = (dm.base_mode == CAOTE_BASE_ACCUM || dm.base_mode == CAOTE_BASE_EXTERNAL) && rt == 0;
  const int tid = threadIdx.x, r = tid >> 4, c0 = tid & 15;
  int n_vis[RPT];
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    const int row = rt * kR + r + 16 * u;
    n_vis[u] = row < dm.R ? n - dm.m + (row % dm.m) + 1 : 0;
  }

  // stage the query tile
  for (int idx = tid; idx < kR * (D / 4); idx += kThreads) {
    const int rr = idx / (D / 4), c4 = idx % (D / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rt * kR + rr < dm.R) v = load4(q + q_offset(dm, b, h, rt * kR + rr) + c4 * 4);
    *reinterpret_cast<float4*>(Qs + rr * LD + c4 * 4) = v;
  }

  const int split_len = ((n + sc.splits - 1) / sc.splits + kKT - 1) / kKT * kKT;
  const int k_begin = split * split_len;
  const int k_end = min(n, k_begin + split_len);
  const T* Ku = K + (size_t)unit * dm.cap * D;
  const T* Vu = V + (size_t)unit * dm.cap * D;

  // l_rest: sum of exp(s - m_run) over the keys so far EXCEPT the first key that sits at the maximum (whose
  // term is exactly 1): the row's 1 - alpha of its top key is then l_rest / (l_rest + 1), a sum of the others
  float m_run[RPT], l_rest[RPT], o_acc[RPT][OC];
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    m_run[u] = -INFINITY;
    l_rest[u] = 0.f;
#pragma unroll
    for (int i = 0; i < OC; ++i) o_acc[u][i] = 0.f;
  }
  float y_acc = 0.f, hb_acc = 0.f;
  constexpr int YP = kThreads / D;  // threads per channel in the base-weighted value sum

  for (int kt = k_begin; kt < k_end; kt += kKT) {
    __syncthreads();
    stage_rows<T, D, LD>(Ks, Ku + (size_t)kt * D, kKT, k_end - kt);
    if (RPT == 1) stage_rows<T, D, LD>(Vs, Vu + (size_t)kt * D, kKT, k_end - kt);
    if (use_base && tid < kKT) bs[tid] = (kt + tid < k_end) ? base[(size_t)unit * dm.cap + kt + tid] : 0.f;
    __syncthreads();

    float s[RPT][4];
    logits<D, LD, RPT>(Qs + r * LD, Ks + c0 * LD, dm.scale, s);  // (rows beyond the length are staged as zeros)
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      float mx = -INFINITY;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = kt + c0 + 16 * i;
        if (j >= k_end || j >= n_vis[u]) s[u][i] = -INFINITY;
        mx = fmaxf(mx, s[u][i]);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(m_run[u], mx);
      const bool new_top = mx > m_run[u];  // this tile holds a key above everything before it
      // (no branch here: the rows of a warp vote together below)
      const float corr = (m_run[u] == -INFINITY) ? 0.f : expf(m_run[u] - m_new);
      float lsum = 0.f;
      bool found = false;  // the first key of the tile at the new maximum (smallest key index) is left out of the sum
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float p = (s[u][i] == -INFINITY) ? 0.f : expf(s[u][i] - m_new);
        if (RPT == 1) Ps[r * kKT + c0 + 16 * i] = p;
        const unsigned at_top = (__ballot_sync(0xffffffffu, new_top && s[u][i] == m_new) >> (threadIdx.x & 16)) & 0xffffu;
        const bool skip = !found && at_top != 0u && (int)(__ffs(at_top) - 1) == c0;
        found |= at_top != 0u;
        lsum += skip ? 0.f : p;
        s[u][i] = p;
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
      // the old top key (term 1 before) joins the others when a new top appears
      l_rest[u] = l_rest[u] * corr + ((new_top && m_run[u] != -INFINITY) ? corr : 0.f) + lsum;
      m_run[u] = m_new;
#pragma unroll
      for (int i = 0; i < OC; ++i) o_acc[u][i] *= corr;
    }
    if constexpr (RPT == 4) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(Ps + (c0 + 16 * i) * kPitch + r * RPT) = make_float4(s[0][i], s[1][i], s[2][i], s[3][i]);
    }
    __syncthreads();
    if (RPT > 1) {
      stage_rows<T, D, LD>(Vs, Vu + (size_t)kt * D, kKT, k_end - kt);
      __syncthreads();
    }

    auto add_key = [&](int j) {
      float p[RPT];
      if constexpr (RPT == 4) *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(Ps + j * kPitch + r * RPT);
      else p[0] = Ps[r * kKT + j];
#pragma unroll
      for (int x = 0; x < OC / 4; ++x) {
        const float4 v = *reinterpret_cast<const float4*>(Vs + j * LD + 64 * x + c0 * 4);
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
          o_acc[u][4 * x] = fmaf(p[u], v.x, o_acc[u][4 * x]);
          o_acc[u][4 * x + 1] = fmaf(p[u], v.y, o_acc[u][4 * x + 1]);
          o_acc[u][4 * x + 2] = fmaf(p[u], v.z, o_acc[u][4 * x + 2]);
          o_acc[u][4 * x + 3] = fmaf(p[u], v.w, o_acc[u][4 * x + 3]);
        }
      }
    };
    // (one row per thread: unrolling and register bound are left to the compiler; larger ones cost 2 - 6 %)
    if constexpr (RPT == 1) {
      for (int j = 0; j < kKT; ++j) add_key(j);
    } else {
#pragma unroll 4
      for (int j = 0; j < kKT; ++j) add_key(j);
    }
    if (use_base) {
      const int col = tid % D, part = tid / D;
      for (int j = part; j < kKT; j += YP) y_acc = fmaf(bs[j], Vs[j * LD + col], y_acc);
      if (tid < kKT) hb_acc += bs[tid];
    }
  }

  const size_t us = (size_t)unit * sc.splits + split;
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    const int row = rt * kR + r + 16 * u;
    if (row < dm.R) {
      if (c0 == 0) {
        sc.part_ml[(us * sc.Rpad + row) * 2 + 0] = m_run[u];
        sc.part_ml[(us * sc.Rpad + row) * 2 + 1] = l_rest[u];
      }
      float* po = sc.part_o + (us * sc.Rpad + row) * D;
#pragma unroll
      for (int x = 0; x < OC / 4; ++x)
        *reinterpret_cast<float4*>(po + 64 * x + c0 * 4) =
            make_float4(o_acc[u][4 * x], o_acc[u][4 * x + 1], o_acc[u][4 * x + 2], o_acc[u][4 * x + 3]);
    }
  }
  if (use_base) {
    __syncthreads();
    red[tid] = y_acc;
    __syncthreads();
    if (tid < D) {
      float y = 0.f;
      for (int p = 0; p < YP; ++p) y += red[p * D + tid];
      sc.part_y[us * D + tid] = y;
    }
    __syncthreads();
    red[tid] = (tid < kKT) ? hb_acc : 0.f;
    __syncthreads();
    if (tid == 0) {
      float hsum = 0.f;
      for (int j = 0; j < kKT; ++j) hsum += red[j];
      sc.part_hb[us] = hsum;
    }
  }
}

// Is row r one of the rows whose attention defines the base score?
__device__ __forceinline__ bool row_counted(const Dims& dm, int r) {
  if (dm.base_mode == CAOTE_BASE_LAST_QUERY) return (r % dm.m) == dm.m - 1;
  return dm.base_mode != CAOTE_BASE_EXTERNAL;
}

// grid = (chunks of rows, units); a thread is a channel of every (kCombineThreads / D)-th row of the chunk. What
// it costs is round trips to L2: the splits' statistics and outputs are fetched eight at a time before the first is used
// (a thread per channel for 32 rows, one value after the other: 27 - 83 us for 28 - 96 rows in up to 32 splits).
template <typename T, int D>
__global__ void __launch_bounds__(kCombineThreads)
attn_combine_kernel(Dims dm, const int* __restrict__ len, Scratch sc, float* __restrict__ o) {
  constexpr int kGroups = kCombineThreads / D, kFly = 8;
  ptx::pdl_wait();
  ptx::pdl_trigger();
  __shared__ float part[kGroups][D];
  const int unit = blockIdx.y, chunk = blockIdx.x, c = threadIdx.x % D, grp = threadIdx.x / D;
  const int b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b];
  if (n == 0 || n < dm.m || n > dm.cap) return;
  float osum = 0.f;
  const int r_end = min(dm.R, (chunk + 1) * sc.chunk_rows);
  for (int r = chunk * sc.chunk_rows + grp; r < r_end; r += kGroups) {
    const float2* ml = reinterpret_cast<const float2*>(sc.part_ml) + (size_t)unit * sc.splits * sc.Rpad + r;
    const float* po = sc.part_o + ((size_t)unit * sc.splits * sc.Rpad + r) * D + c;
    float mx = -INFINITY;
    for (int s0 = 0; s0 < sc.splits; s0 += kFly) {
      float v[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) v[u] = (s0 + u < sc.splits) ? ml[(size_t)(s0 + u) * sc.Rpad].x : -INFINITY;
#pragma unroll
      for (int u = 0; u < kFly; ++u) mx = fmaxf(mx, v[u]);
    }
    float l_rest = 0.f, acc = 0.f;
    bool top_seen = false;  // the first split at the overall maximum keeps its top key apart; the others' join the rest
    for (int s0 = 0; s0 < sc.splits; s0 += kFly) {
      float2 st[kFly];
      float ov[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const bool in = s0 + u < sc.splits;
        st[u] = in ? ml[(size_t)(s0 + u) * sc.Rpad] : make_float2(-INFINITY, 0.f);
        ov[u] = in ? po[(size_t)(s0 + u) * sc.Rpad * D] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        if (st[u].x == -INFINITY) continue;  // (a split in which the row sees no key)
        const float f = expf(st[u].x - mx);
        l_rest = fmaf(st[u].y, f, l_rest);
        if (st[u].x == mx && !top_seen) top_seen = true;
        else l_rest += f;
        acc = fmaf(ov[u], f, acc);
      }
    }
    const float inv_l = 1.f / (l_rest + 1.f);
    const float val = acc * inv_l;
    o[q_offset(dm, b, h, r) + c] = val;
    if (row_counted(dm, r)) osum += val;
    if (c == 0) {
      sc.stats[((size_t)unit * sc.Rpad + r) * 4 + 0] = mx;
      sc.stats[((size_t)unit * sc.Rpad + r) * 4 + 1] = inv_l;
      sc.stats[((size_t)unit * sc.Rpad + r) * 4 + 2] = l_rest * inv_l;
    }
  }
  part[grp][c] = osum;
  __syncthreads();
  if (grp == 0) {
    for (int g = 1; g < kGroups; ++g) osum += part[g][c];
    sc.osum[((size_t)unit * sc.chunks + chunk) * D + c] = osum;
  }
  if (chunk == 0 && grp == kGroups - 1 && (dm.base_mode == CAOTE_BASE_ACCUM || dm.base_mode == CAOTE_BASE_EXTERNAL)) {
    float y = 0.f;
    double hb = 0.0;
    for (int s0 = 0; s0 < sc.splits; s0 += kFly) {
      float yv[kFly], hv[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const size_t us = (size_t)unit * sc.splits + min(s0 + u, sc.splits - 1);
        yv[u] = sc.part_y[us * D + c];
        hv[u] = sc.part_hb[us];
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        if (s0 + u < sc.splits) {
          y += yv[u];
          hb += (double)hv[u];
        }
      }
    }
    sc.ytot[(size_t)unit * D + c] = y;
    if (c == 0) sc.hbtot[unit] = (float)hb;
  }
}

template <typename T, int D, int RPT>
__global__ void __launch_bounds__(kThreads)
score_pass_kernel(Dims dm, const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                  const int* __restrict__ len, float* __restrict__ base, Scratch sc,
                  float* __restrict__ scores, const float* __restrict__ vsum) {
  constexpr int LD = D + 4, kR = kRT * RPT;
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;              // kR * LD
  float* Ks = Qs + kR * LD;      // kKT * LD
  float* Hred = Ks + kKT * LD;   // kRT * kKT  sums of the rows' weights of a key
  float* Cred = Hred + kRT * kKT;  // kRT * kKT  sums of the rows' complements 1 - alpha of a key
  float* Xs = Cred + kRT * kKT;  // D
  float* st = Xs + D;            // kR * 4
  float* wq = st + kR * 4;       // kKT: w_j / (1 - w_j)

  const int unit = blockIdx.y;
  const int b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b];
  const int j0 = blockIdx.x * kKT;
  if (n == 0 || n < dm.m || n > dm.cap || j0 >= n) return;
  const int tid = threadIdx.x, r = tid >> 4, c0 = tid & 15;
  const int mode = dm.base_mode;
  const int n_rows = (mode == CAOTE_BASE_LAST_QUERY) ? dm.G : (mode == CAOTE_BASE_EXTERNAL ? 0 : dm.R);
  const bool carried = (mode == CAOTE_BASE_ACCUM || mode == CAOTE_BASE_EXTERNAL);
  const float hb = carried ? sc.hbtot[unit] : 0.f;
  const float Htot = (float)n_rows + hb;

  // X = (sum of counted output rows + sum_j base_j v_j) / (counted rows + sum_j base_j)
  if (tid < D) {
    float x = 0.f;
    #pragma unroll 8
    for (int ch = 0; ch < sc.chunks; ++ch) x += sc.osum[((size_t)unit * sc.chunks + ch) * D + tid];
    if (carried) x += sc.ytot[(size_t)unit * D + tid];
    Xs[tid] = (Htot > 0.f) ? x / Htot : 0.f;
    if (vsum) Xs[tid] = vsum[(size_t)unit * D + tid] / (float)n;  // FastCAOTE (Sec. 3.3): the mean of the cached values
  }
  const int valid = min(kKT, n - j0);
  if (n_rows > 0) stage_rows<T, D, LD>(Ks, K + ((size_t)unit * dm.cap + j0) * D, kKT, valid);

  // hacc: sum over the counted rows of alpha_{r,j}; cacc: sum of 1 - alpha_{r,j}, where the row's top key takes
  // (sum of the others) / sum from the attention pass and everybody else 1 - alpha <= 1/2: no cancellation
  float hacc[4] = {0.f, 0.f, 0.f, 0.f}, cacc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int t0 = 0; t0 < n_rows; t0 += kR) {
    __syncthreads();
    // counted row number t -> row of the unit
    for (int idx = tid; idx < kR * (D / 4); idx += kThreads) {
      const int rr = idx / (D / 4), c4 = idx % (D / 4);
      const int t = t0 + rr;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (t < n_rows) {
        const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
        v = load4(q + q_offset(dm, b, h, row) + c4 * 4);
      }
      *reinterpret_cast<float4*>(Qs + rr * LD + c4 * 4) = v;
    }
    if (tid < kR) {
      const int t = t0 + tid;
      float mx = 0.f, il = 0.f, cr = 0.f;
      if (t < n_rows) {
        const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
        mx = sc.stats[((size_t)unit * sc.Rpad + row) * 4];
        il = sc.stats[((size_t)unit * sc.Rpad + row) * 4 + 1];
        cr = sc.stats[((size_t)unit * sc.Rpad + row) * 4 + 2];
      }
      st[tid * 4] = mx;
      st[tid * 4 + 1] = il;
      st[tid * 4 + 2] = cr;
    }
    __syncthreads();
    if (t0 + r < n_rows) {
      float s[RPT][4];
      logits<D, LD, RPT>(Qs + r * LD, Ks + c0 * LD, dm.scale, s);
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        const int t = t0 + r + 16 * u;
        if (u > 0 && t >= n_rows) break;
        const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
        const int n_vis = n - dm.m + (row % dm.m) + 1;
        const float mx = st[(r + 16 * u) * 4], il = st[(r + 16 * u) * 4 + 1], cr = st[(r + 16 * u) * 4 + 2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = j0 + c0 + 16 * i;
          if (j < n_vis) {
            const float sl = s[u][i];
            const float a = expf(sl - mx) * il;
            hacc[i] += a;
            cacc[i] += (sl == mx) ? cr : 1.f - a;
          } else {
            cacc[i] += 1.f;  // a row that cannot see the key gives all its weight to the others
          }
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    Hred[r * kKT + c0 + 16 * i] = hacc[i];
    Cred[r * kKT + c0 + 16 * i] = cacc[i];
  }
  __syncthreads();
  if (tid < kKT) {
    const int j = j0 + tid;
    float ratio = 0.f;
    if (j < n) {
      float hj = 0.f, rest = 0.f;  // rest = (1 - w_j) * Htot as a sum of non-negative parts
      for (int rr = 0; rr < kRT; ++rr) {
        hj += Hred[rr * kKT + tid];
        rest += Cred[rr * kKT + tid];
      }
      if (carried) {
        // (the carried scores' own complement is a plain difference: a single carried score that holds almost
        // all of their sum is outside what this any-shape path resolves)
        const float bj = base[(size_t)unit * dm.cap + j];
        rest += hb - bj;
        if (mode == CAOTE_BASE_ACCUM) {
          hj += bj;
          base[(size_t)unit * dm.cap + j] = hj;
        } else {
          hj = bj;
        }
      }
      if (Htot > 0.f && hj > 0.f) ratio = (rest > 0.f) ? hj / rest : INFINITY;
    }
    wq[tid] = ratio;
  }
  __syncthreads();
  // || X - v_j ||: 4 threads per token, D/4 consecutive channels each
  {
    const int key = tid >> 2, part = tid & 3;
    const int j = j0 + key;
    float acc = 0.f;
    if (j < n) {
      const T* vrow = V + ((size_t)unit * dm.cap + j) * D + part * (D / 4);
#pragma unroll
      for (int c = 0; c < D / 4; c += 4) {
        const float4 v = load4(vrow + c);
        const float* x = Xs + part * (D / 4) + c;
        const float d0 = x[0] - v.x, d1 = x[1] - v.y, d2 = x[2] - v.z, d3 = x[3] - v.w;
        acc = fmaf(d0, d0, acc);
        acc = fmaf(d1, d1, acc);
        acc = fmaf(d2, d2, acc);
        acc = fmaf(d3, d3, acc);
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (part == 0 && j < n) {
      const float ratio = wq[key];
      const float nrm = sqrtf(acc);
      // ratio == +inf with a zero distance still means "holds all the weight": keep +inf
      scores[(size_t)unit * dm.cap + j] = (ratio == 0.f) ? 0.f : ((ratio == INFINITY) ? INFINITY : ratio * nrm);
    }
  }
}

inline size_t partial_smem(int D, int rpt) {
  const int LD = D + 4;
  return sizeof(float) * (size_t)(kRT * rpt * LD + (rpt == 1 ? 2 : 1) * kKT * LD + kKT * p_pitch(rpt) + kKT + kThreads);
}
// Sum-of-errors aggregation: instead of adding the rows' weights and applying the general form once,
// add up the exact single-query errors (Theorem 3.2, row by row) of the rows that define the base score:
//     c_j = sum_r alpha_{r,j} / (1 - alpha_{r,j}) * || o_r - v_j ||_2 .
// Needs o and the row statistics of attn_partial / attn_combine. grid = (key tiles, units), kThreads;
// thread (r = tid / 16, c0 = tid % 16) owns row slot r and keys c0 + 16 i of the tile.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
sum_errors_kernel(Dims dm, const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                  const int* __restrict__ len, const float* __restrict__ o, Scratch sc, float* __restrict__ scores) {
  constexpr int LD = D + 4;
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;              // kRT * LD
  float* Os = Qs + kRT * LD;     // kRT * LD
  float* Ks = Os + kRT * LD;     // kKT * LD
  float* Vs = Ks + kKT * LD;     // kKT * LD
  float* Hred = Vs + kKT * LD;   // kRT * kKT
  float* st = Hred + kRT * kKT;  // kRT * 2

  const int unit = blockIdx.y;
  const int b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b];
  const int j0 = blockIdx.x * kKT;
  if (n == 0 || n < dm.m || n > dm.cap || j0 >= n) return;
  const int tid = threadIdx.x, r = tid >> 4, c0 = tid & 15;
  const int mode = dm.base_mode;
  const int n_rows = (mode == CAOTE_BASE_LAST_QUERY) ? dm.G : dm.R;
  const int valid = min(kKT, n - j0);
  stage_rows<T, D, LD>(Ks, K + ((size_t)unit * dm.cap + j0) * D, kKT, valid);
  stage_rows<T, D, LD>(Vs, V + ((size_t)unit * dm.cap + j0) * D, kKT, valid);

  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int t0 = 0; t0 < n_rows; t0 += kRT) {
    __syncthreads();
    for (int idx = tid; idx < kRT * (D / 4); idx += kThreads) {
      const int rr = idx / (D / 4), c4 = idx % (D / 4);
      const int t = t0 + rr;
      float4 qv = make_float4(0.f, 0.f, 0.f, 0.f), ov = qv;
      if (t < n_rows) {
        const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
        qv = load4(q + q_offset(dm, b, h, row) + c4 * 4);
        ov = *reinterpret_cast<const float4*>(o + q_offset(dm, b, h, row) + c4 * 4);
      }
      *reinterpret_cast<float4*>(Qs + rr * LD + c4 * 4) = qv;
      *reinterpret_cast<float4*>(Os + rr * LD + c4 * 4) = ov;
    }
    if (tid < kRT) {
      const int t = t0 + tid;
      float mx = 0.f, il = 0.f, cr = 0.f;
      if (t < n_rows) {
        const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
        mx = sc.stats[((size_t)unit * sc.Rpad + row) * 4];
        il = sc.stats[((size_t)unit * sc.Rpad + row) * 4 + 1];
        cr = sc.stats[((size_t)unit * sc.Rpad + row) * 4 + 2];
      }
      st[tid * 4] = mx;
      st[tid * 4 + 1] = il;
      st[tid * 4 + 2] = cr;
    }
    __syncthreads();
    const int t = t0 + r;
    if (t < n_rows) {
      const int row = (mode == CAOTE_BASE_LAST_QUERY) ? t * dm.m + dm.m - 1 : t;
      const int n_vis = n - dm.m + (row % dm.m) + 1;
      const float mx = st[r * 4], il = st[r * 4 + 1], cr = st[r * 4 + 2];
      float sl4[1][4];
      logits<D, LD, 1>(Qs + r * LD, Ks + c0 * LD, dm.scale, sl4);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int jj = c0 + 16 * i, j = j0 + jj;
        if (j < n_vis) {
          const float sl = sl4[0][i];
          const float e = expf(sl - mx) * il;              // alpha
          const float rest = (sl == mx) ? cr : 1.f - e;    // 1 - alpha: the others' share, without cancellation
          float d2 = 0.f;
#pragma unroll 8
          for (int c = 0; c < D; c += 4) {
            const float4 ov = *reinterpret_cast<const float4*>(Os + r * LD + c);
            const float4 vv = *reinterpret_cast<const float4*>(Vs + jj * LD + c);
            const float a0 = ov.x - vv.x, a1 = ov.y - vv.y, a2 = ov.z - vv.z, a3 = ov.w - vv.w;
            d2 = fmaf(a0, a0, d2); d2 = fmaf(a1, a1, d2); d2 = fmaf(a2, a2, d2); d2 = fmaf(a3, a3, d2);
          }
          acc[i] += (rest > 0.f) ? e / rest * sqrtf(d2) : INFINITY;
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) Hred[r * kKT + c0 + 16 * i] = acc[i];
  __syncthreads();
  if (tid < kKT && j0 + tid < n) {
    float cj = 0.f;
    for (int rr = 0; rr < kRT; ++rr) cj += Hred[rr * kKT + tid];
    scores[(size_t)unit * dm.cap + j0 + tid] = cj;
  }
}

inline size_t sum_errors_smem(int D) {
  const int LD = D + 4;
  return sizeof(float) * (size_t)(2 * kRT * LD + 2 * kKT * LD + kRT * kKT + kRT * 4);
}

inline size_t score_smem(int D, int rpt) {
  const int LD = D + 4;
  return sizeof(float) * (size_t)(kRT * rpt * LD + kKT * LD + 2 * kRT * kKT + D + kRT * rpt * 4 + kKT);
}

}  // namespace generic
}  // namespace caote
