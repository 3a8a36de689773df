// Post-eviction attention output (Sec. 2, budgeted generation; Sec. 3.1, proof of Theorem 3.2): what the
// output of each query row becomes once the evicted tokens are gone and the remaining attention weights
// are renormalised,
//     o'_r = (o_r - sum_{e in E} alpha_{r,e} v_e) / (1 - sum_{e in E} alpha_{r,e}),
// E = the evicted slots the row can see. The weights alpha_{r,e} need the row's softmax normaliser. Where the
// scoring call that ran just before on the same workspace has left the rows' statistics there (the cluster
// decode kernel: one per query head; the tensor-core prefill kernels: one per row; both as reference +
// log2(sum) of the log2-domain logits), they are used and the kernel touches only q, the evicted K / V rows
// and o; the kind of statistics present is a tag in the workspace header. Otherwise the normaliser is
// recomputed with one pass over K (fp32 on the CUDA cores, any dtype, head_dim 64 or 128).
// grid = (ceil(R / kRows), units), 256 threads: one warp per query row.
// Blocks of queries with per-row statistics (the tensor-core row-block kernels) have a tensor-core kernel of their own
// further down, which shares the evicted rows among 128 query rows; this one then leaves those calls alone.
#pragma once

#include "common.cuh"
#include "prefill_tc.cuh"

namespace caote {
namespace post {

constexpr int kRows = 8;
constexpr int kKeys = 64;

template <int D>
inline size_t smem_bytes() { return sizeof(float) * ((size_t)kKeys * (D + 4) + (size_t)kRows * D); }

template <typename T, int D>
__global__ void __launch_bounds__(32 * kRows)
post_evict_kernel(Dims dm, const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                  const int* __restrict__ len, const int* __restrict__ evict_idx, int max_evict,
                  const int* __restrict__ n_evict, const float* __restrict__ o, float* __restrict__ o_post,
                  const int* __restrict__ stat_tag, const float* __restrict__ stats, int prefill_stride,
                  int rows_kernel_ran) {
  constexpr int LD = D + 4, CPL = D / 32;  // channels per lane
  ptx::pdl_wait();
  ptx::pdl_trigger();
  if (rows_kernel_ran && stat_tag && *stat_tag == kStatPerRow) return;  // post_evict_tc_kernel has done the work
  extern __shared__ __align__(16) float smem[];
  float* Ks = smem;             // [kKeys][LD]
  float* Qs = Ks + kKeys * LD;  // [kRows][D]
  const int unit = blockIdx.y, b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b], m = dm.m;
  if (n <= 0 || n < m || n > dm.cap) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x * kRows + warp;
  const bool row_ok = r < dm.R;
  const int g = row_ok ? r / m : 0, i = row_ok ? r % m : 0;
  const size_t qoff = (((size_t)b * dm.Hq + h * dm.G + g) * m + i) * D;
  const int n_vis = row_ok ? n - m + i + 1 : 0;
  for (int c = lane; c < D; c += 32) Qs[warp * D + c] = row_ok ? to_float(q[qoff + c]) : 0.f;
  const T* Ku = K + (size_t)unit * dm.cap * D;
  const T* Vu = V + (size_t)unit * dm.cap * D;

  // statistics left by the scoring call? (1: per query head, 2: per row; anything else: none)
  const int tag = stat_tag ? *stat_tag : 0;
  const bool have_stat = (tag == kStatPerHead && m == 1) || tag == kStatPerRow;
  float stat2 = 0.f;  // alpha = 2^(log2(e) * scale * <q, k> - stat2)
  if (have_stat && row_ok)
    stat2 = (tag == kStatPerHead) ? stats[(size_t)unit * kHeadStatFloats + g] : -stats[(size_t)unit * prefill_stride + r];  // (the row blocks leave it negated)
  // pass over the keys: running maximum and sum of exp of this row's logits, two keys per lane and tile
  float mx = -INFINITY, l = 0.f;
  for (int kt = 0; kt < (have_stat ? 0 : n); kt += kKeys) {
    __syncthreads();
    for (int idx = tid; idx < kKeys * (D / 4); idx += blockDim.x) {
      const int rr = idx / (D / 4), c4 = idx % (D / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kt + rr < n) v = load4(Ku + (size_t)(kt + rr) * D + c4 * 4);
      *reinterpret_cast<float4*>(Ks + rr * LD + c4 * 4) = v;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int jj = lane + 32 * t, j = kt + jj;
      if (j < n_vis) {
        float s = 0.f;
#pragma unroll 8
        for (int c = 0; c < D; c += 4) {
          const float4 kv = *reinterpret_cast<const float4*>(Ks + jj * LD + c);
          const float4 qv = *reinterpret_cast<const float4*>(Qs + warp * D + c);
          s = fmaf(qv.x, kv.x, s); s = fmaf(qv.y, kv.y, s); s = fmaf(qv.z, kv.z, s); s = fmaf(qv.w, kv.w, s);
        }
        s *= dm.scale;
        const float nm = fmaxf(mx, s);
        l = l * __expf(mx - nm) + __expf(s - nm);
        mx = nm;
      }
    }
  }
  const float M = warp_max(mx);
  const float Z = warp_sum(mx == -INFINITY ? 0.f : l * __expf(mx - M));
  if (!row_ok) return;

  // the evicted slots this row sees: their weights and weighted values (lane = CPL channels)
  const int k = n_evict[b];
  const int* E = evict_idx + (size_t)unit * max_evict;
  float A = 0.f, Y[CPL];
  int left = n_vis;  // tokens the row still sees: where none is left the output is 0, whatever 1 - A rounds to
#pragma unroll
  for (int c = 0; c < CPL; ++c) Y[c] = 0.f;
  for (int e = 0; e < k; ++e) {
    const int j = E[e];
    if (j < 0 || j >= n_vis) continue;
    --left;
    float part = 0.f, vv[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      part = fmaf(Qs[warp * D + lane * CPL + c], to_float(Ku[(size_t)j * D + lane * CPL + c]), part);
      vv[c] = to_float(Vu[(size_t)j * D + lane * CPL + c]);
    }
    const float s = warp_sum(part) * dm.scale;
    const float a = have_stat ? exp2f(s * 1.4426950408889634f - stat2) : __expf(s - M) / Z;
    A += a;
#pragma unroll
    for (int c = 0; c < CPL; ++c) Y[c] = fmaf(a, vv[c], Y[c]);
  }
  const float rest = 1.f - A;
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const size_t at = qoff + lane * CPL + c;
    o_post[at] = rest > 0.f && left > 0 ? (o[at] - Y[c]) / rest : 0.f;
  }
}

// The same correction for blocks of queries whose rows' statistics the scoring call left behind (bf16): does nothing
// unless the workspace header says so. It is the attention pass over the evicted rows with a reference that is already
// known, so a CTA takes 128 query rows of a unit (two threads per row) and walks the unit's evicted slots 128 at a time:
// their K and V rows are gathered into swizzled tiles by plain loads, S = Q K_E^T and Y += P V_E (P as two bf16 parts) run
// on tcgen05, and the weights 2^(s + stat) are formed in between. What bounds it is the chain of one tile (gather, product,
// exponentials, product, write-out): 16 units x 896 rows x 128 evictions, 82 us on the CUDA cores (a CTA per 16 rows) -> 25 between events.
// grid = (ceil(R / 128), units), 256 threads; TMEM columns: S / P [0, 128), Y [128, 128 + D).
constexpr int kTcThreads = 256;
template <int D>
inline size_t tc_smem_bytes() {
  return 1024 + 3 * (size_t)prefill::kTileBytesOf<D> + prefill::kTile * sizeof(int) + kTcThreads * (sizeof(float) + sizeof(int)) + 64;
}

template <int D>
__global__ void __launch_bounds__(kTcThreads, 2)
post_evict_tc_kernel(Dims dm, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ K,
                     const __nv_bfloat16* __restrict__ V, const int* __restrict__ len, const int* __restrict__ evict_idx,
                     int max_evict, const int* __restrict__ n_evict, const float* o, float* o_post,
                     const int* __restrict__ stat_tag, const float* __restrict__ stats, int stat_stride, int* status) {
  using namespace prefill;
  constexpr int kTB = kTileBytesOf<D>, kChunks = D / 8;  // 16-byte chunks of a row
  ptx::pdl_wait();
  ptx::pdl_trigger();
  if (*stat_tag != kStatPerRow) return;
  extern __shared__ char smem_raw[];
  char* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  char *Qs = sm, *Ks = Qs + kTB, *Vs = Ks + kTB;
  int* js = reinterpret_cast<int*>(Vs + kTB);               // [kTile] slot of the evicted token, -1: none
  float* xa = reinterpret_cast<float*>(js + kTile);         // [kTcThreads] half rows' sums of weights,
  int* xg = reinterpret_cast<int*>(xa + kTcThreads);        // [kTcThreads] and numbers of evicted tokens
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(xg + kTcThreads);
  uint64_t* y_bar = s_bar + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(y_bar + 1);

  const int unit = blockIdx.y, b = unit / dm.Hkv;
  const int n = len[b], m = dm.m, k = n_evict[b];
  if (n <= 0 || n < m || n > dm.cap) return;
  const int tid = threadIdx.x, warp = ptx::warp_index(), r0 = blockIdx.x * kTile;
  const int half = tid >> 7, r = r0 + (tid & (kTile - 1));
  const __nv_bfloat16* Ku = K + (size_t)unit * dm.cap * D;
  const __nv_bfloat16* Vu = V + (size_t)unit * dm.cap * D;
  const int* E = evict_idx + (size_t)unit * max_evict;
  if (tid == 0) {
    mbar_init(s_bar, 1);
    mbar_init(y_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tmem_slot, 256);
  for (int idx = tid; idx < kTile * kChunks; idx += kTcThreads) {
    const int rr = idx / kChunks, c = idx % kChunks;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r0 + rr < dm.R) v = *reinterpret_cast<const uint4*>(q + ((size_t)unit * dm.R + r0 + rr) * D + 8 * c);
    *reinterpret_cast<uint4*>(Qs + ptx::tile_off(rr, c)) = v;
  }
  const float stat = (r < dm.R) ? stats[(size_t)unit * stat_stride + r] : -INFINITY;  // (negated there; rows beyond R: weights 0)
  const int n_vis = (r < dm.R) ? n - m + (r % m) + 1 : 0;
  const float scale2 = dm.scale * 1.4426950408889634f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot, t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  float A = 0.f;
  int gone = 0, t = 0;  // gone: evicted tokens that the row sees, in this thread's half
  for (int e0 = 0; e0 < k; e0 += kTile, ++t) {
    if (t > 0) mbar_wait(y_bar, (t - 1) & 1, status);  // the tiles of the evicted rows have been read
    if (tid < kTile) {
      int j = (e0 + tid < k) ? E[e0 + tid] : -1;
      js[tid] = (j >= 0 && j < n) ? j : -1;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTile * kChunks / kTcThreads; ++i) {
      const int idx = tid + i * kTcThreads, e = idx / kChunks, c = idx % kChunks, j = js[e];
      uint4 kr = make_uint4(0u, 0u, 0u, 0u), vr = kr;
      if (j >= 0) {
        kr = *reinterpret_cast<const uint4*>(Ku + (size_t)j * D + 8 * c);
        vr = *reinterpret_cast<const uint4*>(Vu + (size_t)j * D + 8 * c);
      }
      *reinterpret_cast<uint4*>(Ks + ptx::tile_off(e, c)) = kr;
      *reinterpret_cast<uint4*>(Vs + ptx::tile_off(e, c)) = vr;
    }
    fence_async_smem();
    __syncthreads();
    if (warp == 0 && ptx::elect_one()) {
      tc_fence_after();
      const uint64_t qd = smem_desc(smem_u32(Qs), 16, 1024), kd = smem_desc(smem_u32(Ks), 16, 1024);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) umma(tmem, qd + k_major_step(ks), kd + k_major_step(ks), instr_desc_n(false, kTile), ks > 0);
      umma_commit(s_bar);
    }
    mbar_wait(s_bar, t & 1, status);
    tc_fence_after();
    float sv[64];
    tmem_ld32(t_lane + half * 64, *reinterpret_cast<float(*)[32]>(&sv[0]));
    tmem_ld32(t_lane + half * 64 + 32, *reinterpret_cast<float(*)[32]>(&sv[32]));
    uint32_t hi[32], lo[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const int2 jj = *reinterpret_cast<const int2*>(js + half * 64 + 2 * c);
      const bool v0 = jj.x >= 0 && jj.x < n_vis, v1 = jj.y >= 0 && jj.y < n_vis;
      const float p0 = v0 ? fast_exp2(fmaf(sv[2 * c], scale2, stat)) : 0.f;
      const float p1 = v1 ? fast_exp2(fmaf(sv[2 * c + 1], scale2, stat)) : 0.f;
      gone += (v0 ? 1 : 0) + (v1 ? 1 : 0);
      const uint32_t b0 = __float_as_uint(p0), b1 = __float_as_uint(p1);
      hi[c] = __byte_perm(b0, b1, 0x7632);
      lo[c] = pack_bf16(p0 - __uint_as_float(b0 & 0xffff0000u), p1 - __uint_as_float(b1 & 0xffff0000u));
      A += p0 + p1;
    }
    tc_fence_before();
    __syncthreads();  // both halves of every row have read their S columns
    tc_fence_after();
    tmem_st32u(t_lane + half * 32, hi);
    tmem_st32u(t_lane + 64 + half * 32, lo);
    tmem_st_wait();
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && ptx::elect_one()) {
      tc_fence_after();
      constexpr uint32_t kIdesc = instr_desc_n(true, D);
      const uint64_t vd = smem_desc(smem_u32(Vs), kHalfBytes, 1024);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        umma_ts(tmem + kTile, tmem + ks * 8, vd + mn_major_step(ks), kIdesc, t > 0 || ks > 0);
        umma_ts(tmem + kTile, tmem + 64 + ks * 8, vd + mn_major_step(ks), kIdesc, true);
      }
      umma_commit(y_bar);
    }
  }
  xa[tid] = A;
  xg[tid] = gone;
  __syncthreads();
  // (where the row sees none of the retained tokens its output is 0, whatever 1 - A rounds to)
  const float rest = xg[tid] + xg[tid ^ kTile] < n_vis ? 1.f - (xa[tid] + xa[tid ^ kTile]) : 0.f;
  if (t > 0) mbar_wait(y_bar, (t - 1) & 1, status);
  tc_fence_after();
#pragma unroll
  for (int cc = 0; cc < D / 64; ++cc) {
    const int c0 = half * (D / 2) + cc * 32;
    float y[32];
    if (t > 0) {
      tmem_ld32(t_lane + kTile + c0, y);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) y[i] = 0.f;
    }
    if (r < dm.R) {
      const size_t at = ((size_t)unit * dm.R + r) * D + c0;
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 o4 = *reinterpret_cast<const float4*>(o + at + i);
        float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rest > 0.f) res = make_float4((o4.x - y[i]) / rest, (o4.y - y[i + 1]) / rest, (o4.z - y[i + 2]) / rest, (o4.w - y[i + 3]) / rest);
        *reinterpret_cast<float4*>(o_post + at + i) = res;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 256);
}

}  // namespace post
}  // namespace caote
