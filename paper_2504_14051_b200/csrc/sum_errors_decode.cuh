// Sum-of-errors aggregation for a single query per head (bf16, up to 8 query heads per KV head): the score of a cached
// token is the sum over the group's heads of the exact single-head eviction error (Sec. 3.1, Theorem 3.2),
//     c_j = sum_g alpha_{g,j} / (1 - alpha_{g,j}) * || o_g - v_j ||_2 .
// It runs after the cluster kernel, which has written the heads' outputs o_g and left per head the log-sum-exp m_g
// (alpha_{g,j} = 2^(s_{g,j} - m_g)), the largest logit and the share of all other tokens next to the token that
// holds it. This pass reads K and V once more: logits as matrix products (16 tokens x 8 heads x 16 channels; bf16 operands,
// fp32 sums, as in the attention pass), distances by plain subtraction (no ||o||^2 - 2 o.v + ||v||^2: for a token that
// holds nearly all of a head's weight o_g is nearly v_j, and a bf16 cross term from the tensor cores would leave nothing of
// the difference). 1 - alpha of a head's top token is the stored share of the others, never a difference of nearly equal
// numbers.
//
// What bounds it: for one or two heads HBM; from there on the distances, two fp32 operations per (token, head, channel),
// and the latencies in each warp's chain of copy, products, weights, distances. So a CTA takes a run of a unit's tokens, a
// warp takes tiles of it, fills a ring of its own by TMA and handles all of the group's heads (a row is unpacked once), and
// as many warps as fit run side by side. Rings are per warp because loads finish in any order: with stages that pass from
// warp to warp, a warp could wait for a phase while the phase before, another warp's load, is not over, and take the one
// for the other. Measured at 7 heads of 128 channels, 96 units of 3 000 tokens: one tile of 128 tokens per CTA, copied and
// then computed, the heads dealt to four warps, 75 us; pipelined, with the logits on the CUDA cores too, 54; as it is 44. At 64
// units of 16 000 tokens, 0.5 GB: 158 and 127. 96 units, one head: 54, at the rate of a plain copy.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace caote {
namespace sed {

constexpr int kWarps = 4, kThreads = kWarps * 32;
constexpr int kWPitch = 9;  // floats per token of the table of weights (odd: lanes on different banks)
constexpr long long kDrainCycles = 4000000000LL;  // waits at the end for copies that are still in flight after one that ran out

// Tiles by the group's size. Small copies and many warps hide latencies, large copies carry more bytes: 64 (128) units of
// 16 000 tokens, head_dim 128: one head 164 us with large ones, 302 with small ones; 7 heads 133 and 128, 8 heads (128
// units) 278 and 259; 4 heads of 64 channels 135 and 115.
template <int G>
struct Tile {
  static constexpr bool kLarge = G <= 2;
  static constexpr int kTok = kLarge ? 2 : 1, kT = 32 * kTok;  // tokens per lane and per tile of a warp
  static constexpr int kBoxCh = kLarge ? 64 : 32;              // channels of a copy
  static constexpr int kStageBytes = kT * kBoxCh * 2, kStages = (kLarge ? 24 : 10) * 1024 / kStageBytes;  // per warp
  static constexpr int kCtasPerSm = kLarge ? 2 : 4;
};
template <int G, int D>
constexpr size_t smem_bytes_of = 1024 + (size_t)kWarps * Tile<G>::kStages * (Tile<G>::kStageBytes + 8) +
                                 sizeof(float) * (8 * D + 24 + kWarps * Tile<G>::kT * kWPitch);

// CTAs per unit: the fewest rounds of tiles (and one for a CTA's start) over the waves of CTAs.
inline int splits(int units, int cap, int tile, int ctas_per_sm) {
  const int rounds = (cap + tile * kWarps - 1) / (tile * kWarps), wave = ctas_per_sm * g_sm_count;
  int best = 1;
  long long cost = -1;
  for (int s = 1; s <= rounds && s <= 256; ++s) {
    const long long c = (((long long)units * s + wave - 1) / wave) * ((rounds + s - 1) / s + 1);
    if (cost < 0 || c < cost) { cost = c; best = s; }
  }
  return best;
}

// Bounded wait; the first one that runs out says so, and no later wait of the thread blocks (all indices stay in bounds). A
// lane 0 that is late starts no more copies and waits at the end for those it has started.
__device__ __forceinline__ void wait(uint64_t* bar, uint32_t parity, bool& late, int* status, long long limit) {
  if (late || ptx::mbar_try_wait(bar, parity)) return;
  const long long t0 = clock64();
  while (!ptx::mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) {
      set_status(status, CAOTE_ERR_TIMEOUT);
      late = true;
      return;
    }
  }
}

// 16-byte chunk c of row r of a box: rows of 128 (64) bytes, swizzled over their length
template <int kBoxCh>
__device__ __forceinline__ uint32_t box_off(int r, int c) {
  return kBoxCh == 64 ? (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)) : (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&a)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// grid = (splits, units)
template <int G, int D>
__global__ void __launch_bounds__(kThreads, Tile<G>::kCtasPerSm)
sum_errors_decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, Dims dm,
                         const __nv_bfloat16* __restrict__ q, const int* __restrict__ len, const float* __restrict__ o,
                         const float* __restrict__ head_stats, float* __restrict__ scores, int* status,
                         long long wait_cycles) {
  constexpr int kTok = Tile<G>::kTok, kT = Tile<G>::kT, kBoxCh = Tile<G>::kBoxCh, kStageBytes = Tile<G>::kStageBytes,
                kStages = Tile<G>::kStages;
  constexpr int kBoxes = D / kBoxCh, kSubs = 2 * kBoxes;  // stages of a tile: its K boxes, then its V boxes
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ char smem_raw[];
  // (1024-byte alignment by an offset into the array, not by a round trip through an integer: the pointer keeps its
  // address space, so what is read through it compiles to shared-memory loads, not generic ones)
  char* rings = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);      // [warp][stage]
  float* Os = reinterpret_cast<float*>(rings + kWarps * kStages * kStageBytes);  // [8][D], the heads' outputs negated
  float* St = Os + 8 * D;                                                        // [3][8]
  float* Ws = St + 24;                                                           // [warp][kT][kWPitch] weights alpha / (1 - alpha)
  uint64_t* bars = reinterpret_cast<uint64_t*>(Ws + kWarps * kT * kWPitch);      // [warp][stage]

  const int unit = blockIdx.y, b = unit / dm.Hkv, h = unit % dm.Hkv;
  const int n = len[b], tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (n <= 0 || n > dm.cap) return;
  const int nt = (n + kT - 1) / kT, rounds = (nt + kWarps - 1) / kWarps, per = (rounds + (int)gridDim.x - 1) / (int)gridDim.x * kWarps;
  const int t0 = blockIdx.x * per, t1 = min(nt, t0 + per);
  if (t0 >= t1) return;

  // Every warp has a ring of its own, which its lane 0 fills: stage i of the warp is the i-th box of its tiles.
  char* ring = rings + warp * kStages * kStageBytes;
  uint64_t* full = bars + warp * kStages;
  const int mine = t0 + warp < t1 ? (t1 - t0 - warp + kWarps - 1) / kWarps : 0, boxes = mine * kSubs;
  auto load = [&](int i) {
    const int st = i % kStages, sub = i % kSubs, t = t0 + warp + i / kSubs * kWarps;
    ptx::mbar_expect_tx(&full[st], kStageBytes);
    ptx::tma_load_2d(ring + st * kStageBytes, sub < kBoxes ? &tmK : &tmV, kBoxCh * (sub % kBoxes), unit * dm.cap + t * kT, &full[st]);
  };
  if (lane == 0) {
    for (int i = 0; i < kStages; ++i) ptx::mbar_init(&full[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < kStages && i < boxes; ++i) load(i);
  }
  const size_t qo = ((size_t)b * dm.Hq + (size_t)h * G) * D;
  for (int i = tid; i < G * D; i += kThreads) Os[i] = -o[qo + i];  // (negated: the distance pass forms v - o with a packed add)
  if (tid < 24) St[tid] = head_stats[(size_t)unit * kHeadStatFloats + tid];
  // q as the products' second operand: lane l holds channels 2 (l % 4) + {0, 1, 8, 9} of every 16 of head l / 4
  uint32_t qf[D / 16][2];
  const int gh = lane >> 2, gc = 2 * (lane & 3);
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks)
#pragma unroll
    for (int e = 0; e < 2; ++e)
      qf[ks][e] = gh < G ? *reinterpret_cast<const uint32_t*>(q + qo + gh * D + 16 * ks + 8 * e + gc) : 0u;
  __syncthreads();

  const float scale2 = dm.scale * 1.4426950408889634f;
  float* W = Ws + warp * kT * kWPitch;
  bool late = false;
  int i = 0, started = min(kStages, boxes);  // the box that is read, copies started (lane 0)
  auto next = [&]() {  // the stage has been read: the box that takes its place
    ptx::fence_async_smem();  // (by every lane: nothing else keeps the copy behind loads that are still on their way)
    __syncwarp();
    if (lane == 0 && !late && i + kStages < boxes) {
      load(i + kStages);
      ++started;
    }
    ++i;
  };
  for (int t = t0 + warp; t < t1; t += kWarps) {
    // ---- logits (16 tokens x 8 heads per product) and weights ----
    float s[kT / 16][4];
#pragma unroll
    for (int mt = 0; mt < kT / 16; ++mt)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[mt][e] = 0.f;
#pragma unroll
    for (int sub = 0; sub < kBoxes; ++sub) {
      wait(&full[i % kStages], (i / kStages) & 1, late, status, wait_cycles);
      const uint32_t sm = ptx::smem_u32(ring + (i % kStages) * kStageBytes);
#pragma unroll
      for (int ks = 0; ks < kBoxCh / 16; ++ks)
#pragma unroll
        for (int mt = 0; mt < kT / 16; ++mt) {
          uint32_t a[4];
          ldmatrix_x4(sm + box_off<kBoxCh>(16 * mt + (lane & 15), 2 * ks + (lane >> 4)), a);
          mma_bf16(s[mt], a, qf[sub * (kBoxCh / 16) + ks][0], qf[sub * (kBoxCh / 16) + ks][1]);
        }
      next();
    }
#pragma unroll
    for (int mt = 0; mt < kT / 16; ++mt)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int tok = 16 * mt + (lane >> 2) + 8 * (e >> 1), g = gc + (e & 1);
        const float s2 = s[mt][e] * scale2, a = exp2f(s2 - St[g]);
        // the head's top token (its logit, formed here in another order than in the attention pass, within 3e-4 of the
        // largest): the others' share as stored; two tokens that close to the top have weights that close to each other
        const float rest = (s2 >= St[8 + g] - 3e-4f) ? St[16 + g] : 1.f - a;
        if (g < G) W[tok * kWPitch + g] = (a == 0.f) ? 0.f : ((rest > 0.f) ? a / rest : INFINITY);
      }
    // ---- distances: pairs of partial sums over the even and the odd channels (packed fp32 math) ----
    float2 d2[kTok][G];
#pragma unroll
    for (int k = 0; k < kTok; ++k)
#pragma unroll
      for (int g = 0; g < G; ++g) d2[k][g] = make_float2(0.f, 0.f);
#pragma unroll
    for (int sub = 0; sub < kBoxes; ++sub) {
      wait(&full[i % kStages], (i / kStages) & 1, late, status, wait_cycles);
      const char* sm = ring + (i % kStages) * kStageBytes;
      const float* tab = Os + kBoxCh * sub;
#pragma unroll 2
      for (int c = 0; c < kBoxCh / 8; ++c) {  // chunks of 8 channels
        float2 x[kTok][4];
#pragma unroll
        for (int k = 0; k < kTok; ++k) {
          const uint4 raw = *reinterpret_cast<const uint4*>(sm + box_off<kBoxCh>(lane + 32 * k, c));
          const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) x[k][e] = make_float2(__uint_as_float(w4[e] << 16), __uint_as_float(w4[e] & 0xffff0000u));
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float4 y0 = *reinterpret_cast<const float4*>(tab + g * D + 8 * c), y1 = *reinterpret_cast<const float4*>(tab + g * D + 8 * c + 4);
          const float2 y[4] = {make_float2(y0.x, y0.y), make_float2(y0.z, y0.w), make_float2(y1.x, y1.y), make_float2(y1.z, y1.w)};
#pragma unroll
          for (int k = 0; k < kTok; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 df = __fadd2_rn(x[k][e], y[e]);
              d2[k][g] = __ffma2_rn(df, df, d2[k][g]);
            }
        }
      }
      next();
    }
#pragma unroll
    for (int k = 0; k < kTok; ++k) {
      float cj = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float w = W[(lane + 32 * k) * kWPitch + g];
        cj += (w == INFINITY) ? w : w * sqrtf(d2[k][g].x + d2[k][g].y);
      }
      const int j = t * kT + lane + 32 * k;
      if (j < n) scores[(size_t)unit * dm.cap + j] = cj;
    }
    __syncwarp();  // the weights have been read
  }
  if (lane == 0 && late) {  // (nothing may still be on its way to this CTA's shared memory when it ends)
    bool never = false;
    for (int k = max(0, started - kStages); k < started; ++k) wait(&full[k % kStages], (k / kStages) & 1, never, status, kDrainCycles);
  }
}

}  // namespace sed
}  // namespace caote
