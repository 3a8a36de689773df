// FastCAOTE (Sec. 3.3): the CAOTE score with X replaced by the plain mean of the cached values. The mean
// does not depend on this call's attention, so it can be carried from step to step: the library keeps
// vsum[u, :] = sum over the unit's valid slots of V[u, j, :] (fp32) and divides by n when it scores.
//   vsum_kernel        from scratch (one read of V)
//   vsum_add_kernel    += the m rows about to be appended
//   vsum_sub_unit      -= the rows about to be evicted (device function, used by the compaction kernels)
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace caote {
namespace fast {

// One cluster of kSumCtas CTAs per unit, every CTA a contiguous share of its rows; 256 threads, a thread sums one 16-byte
// piece of every (256 / pieces)-th row, four rows in flight; the shares meet in rank 0 in a fixed order. (One CTA per unit
// and two bytes per load: 286 us for 16 units of 6.3 k tokens.)
// kWide: V is 16-byte aligned; where it is not (this call has no rule for it) a piece comes element by element.
constexpr int kSumCtas = 8;
template <typename T, bool kWide>
__device__ __forceinline__ uint4 load_piece(const T* p) {
  if constexpr (kWide) {
    return *reinterpret_cast<const uint4*>(p);
  } else {
    uint32_t w[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if constexpr (sizeof(T) == 2)
        w[c] = (uint32_t)__bfloat16_as_ushort(p[2 * c]) | ((uint32_t)__bfloat16_as_ushort(p[2 * c + 1]) << 16);
      else
        w[c] = __float_as_uint(p[c]);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
}
template <typename T, int D, bool kWide>
__global__ void __launch_bounds__(256)
vsum_kernel(int Hkv, int cap, const T* __restrict__ V, const int* __restrict__ len, float* __restrict__ vsum) {
  constexpr int E = 16 / (int)sizeof(T), P = D / E, kRowsPass = 256 / P, kFly = 4;
  __shared__ float part[kRowsPass][D], mine[D];
  ptx::pdl_wait();
  ptx::pdl_trigger();
  const int unit = blockIdx.x / kSumCtas, rank = (int)ptx::cluster_ctarank(), n = len[unit / Hkv];
  const int piece = threadIdx.x % P, g = threadIdx.x / P;
  const int share = (max(n, 0) + kSumCtas - 1) / kSumCtas, r1 = (n <= cap) ? min(n, (rank + 1) * share) : 0;
  float acc[E];
#pragma unroll
  for (int e = 0; e < E; ++e) acc[e] = 0.f;
  const T* src = V + (size_t)unit * cap * D + piece * E;
  for (int j0 = rank * share + g; j0 < r1; j0 += kFly * kRowsPass) {
    uint4 raw[kFly];
#pragma unroll
    for (int u = 0; u < kFly; ++u)
      raw[u] = (j0 + u * kRowsPass < r1) ? load_piece<T, kWide>(src + (size_t)(j0 + u * kRowsPass) * D) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if constexpr (sizeof(T) == 2) {
          acc[2 * c] += __uint_as_float(w[c] << 16);
          acc[2 * c + 1] += __uint_as_float(w[c] & 0xffff0000u);
        } else {
          acc[c] += __uint_as_float(w[c]);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e) part[g][piece * E + e] = acc[e];
  __syncthreads();
  if (threadIdx.x < D) {
    float s = 0.f;
    for (int r = 0; r < kRowsPass; ++r) s += part[r][threadIdx.x];
    mine[threadIdx.x] = s;
  }
  ptx::cluster_sync_all();
  if (rank == 0 && threadIdx.x < D) {
    float s = 0.f;
    for (int r = 0; r < kSumCtas; ++r) s += ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(mine + threadIdx.x), r));
    vsum[(size_t)unit * D + threadIdx.x] = s;
  }
  ptx::cluster_sync_all();  // (nobody leaves while its share is read)
}

// grid = units, D threads. A sequence that caote_append will skip (no room for m rows) is skipped here too.
template <typename T>
__global__ void vsum_add_kernel(int Hkv, int cap, int m, int D, const T* __restrict__ v_new, const int* __restrict__ len,
                                float* __restrict__ vsum) {
  ptx::pdl_wait();
  ptx::pdl_trigger();
  const int unit = blockIdx.x, n = len[unit / Hkv], c = threadIdx.x;
  if (n < 0 || n + m > cap) return;
  float acc = 0.f;
#pragma unroll 16
  for (int i = 0; i < m; ++i) acc += to_float(v_new[((size_t)unit * m + i) * D + c]);
  vsum[(size_t)unit * D + c] += acc;
}

// The rows listed in evict_idx[unit, 0..k) leave the sum; called by all threads of the unit's CTA before
// the rows are overwritten.
template <typename T>
__device__ inline void vsum_sub_unit(int unit, int k, int cap, int D, const T* __restrict__ V, const int* E,
                                     float* __restrict__ vsum) {  // (E: global or shared memory, possibly written by this CTA)
  for (int c = threadIdx.x; c < D; c += blockDim.x) {
    float acc = 0.f;
#pragma unroll 8
    for (int r = 0; r < k; ++r) acc += to_float(V[((size_t)unit * cap + E[r]) * D + c]);
    vsum[(size_t)unit * D + c] -= acc;
  }
}

// grid = units, 128 threads (the unfused selection / compaction path).
template <typename T>
__global__ void vsum_sub_kernel(int Hkv, int cap, int D, const T* __restrict__ V, const int* __restrict__ evict_idx,
                                int max_evict, const int* __restrict__ n_evict, float* __restrict__ vsum) {
  ptx::pdl_wait();
  ptx::pdl_trigger();
  const int unit = blockIdx.x, k = n_evict[unit / Hkv];
  if (k > 0) vsum_sub_unit<T>(unit, k, cap, D, V, evict_idx + (size_t)unit * max_evict, vsum);
}

}  // namespace fast
}  // namespace caote
