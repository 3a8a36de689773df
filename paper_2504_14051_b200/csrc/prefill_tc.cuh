// Tensor-core scoring path (tcgen05 + TMEM) for bf16, head_dim 64 or 128, any base mode: M = G * m query rows per
// (sequence, KV head) unit against its n cached keys. Blocks of a prompt are what it is built for; it also takes the
// single-query shapes that the cluster kernel has no form for (see decode_shape_ok): a row block is then mostly
// padding, but a pass over K and V at this kernel's pace per tile still keeps up with HBM.
//
//   attn_kernel   rows x keys. One CTA owns 128 query rows of a unit and walks the unit's keys in
//                 tiles of 128: S = Q K^T (tcgen05.mma, fp32 accumulator in TMEM), per-row online
//                 softmax straight out of TMEM (two threads per row, 64 keys each), P back into TMEM
//                 as two bf16 parts (hi + lo, 16 significant bits together), O += P V with P as the
//                 TMEM-side A operand and V as the MN-major B operand. One lane each of three extra warps
//                 issues the products, the K copies and the V copies, so the tensor pipe always has the
//                 next S queued while the rows are busy with the current one. Few row blocks leave SMs idle: the
//                 keys of a unit are then split among the CTAs of a thread-block cluster, which merge their
//                 outputs and statistics through distributed shared memory. Writes o, the per-row softmax
//                 statistics (reference + log2 of the sum) and, per CTA, the sum of its counted rows: all for
//                 CHUNK_SUM and ACCUM, the last of every head for LAST_QUERY, none for EXTERNAL.
//   carried_sum_kernel  (ACCUM, EXTERNAL) parts of sum_j base_j v_j and sum_j base_j. It needs nothing of the attention
//                 pass, so as its dependent launch it does its work on the SMs that one leaves free or is done with,
//                 and only then waits for it.
//                 X = sum_j w_j v_j = (sum of the counted output rows + sum_j base_j v_j) / (counted rows + sum_j base_j).
//   score_kernel  keys x counted rows. One CTA owns 256 keys of a unit (two key tiles) and walks the unit's
//                 counted rows in blocks of 128: S^T = K Q^T lands in TMEM with one key per lane, so each
//                 thread sums exp2(s - ref_r) / sum_r over the rows of its own key without any
//                 exchange: h_j = sum_r alpha_{r,j} (+ base_j). Then c_j = w_j / (1 - w_j) * ||X - v_j||, X from its parts.
//
//   dominant_kernel  (all but EXTERNAL) scores the token that holds most of a unit's weight again, if there is one.
//
// 1 - w_j. With 64 counted rows or more it is formed as the difference H - h_j of the sum of all weights (rows, and carried
// scores) and the token's own, both good to about 1e-6 of H: a weight of a few thousand exponentials, each with the rounding of
// its statistic (|stat| 6e-8) and a quarter of them from a polynomial (3e-6, of alternating sign). For fewer rows (`few`) the
// attention pass keeps the largest numerator of every counted row apart from the sum of the others, and the complement of
// the row's top token is that sum's share, everybody else's 1 - alpha with alpha <= 1/2. Either is enough as long as nobody
// holds most of the weight. For a token that does (an attention sink), || X - v_j || suffers as well: X is nearly v_j, and the
// tensor pipe's running sums lose about 1e-6 of it towards zero, so at 1 - w_j = 1e-4 the score was 7e-3 off. There is at most one
// token above kDominant of H; dominant_kernel forms its complement as the sum of the others' weights and its distance
// as || sum_i w_i (v_i - v_j) || over the others: nothing cancels.
//
// Operands are staged by TMA as 64-channel boxes with the 128-byte swizzle, which is the canonical
// K-major UMMA layout (8-row groups 1024 bytes apart); V in the second product is read through an
// MN-major descriptor of the same bytes. Every mbarrier wait is bounded by a clock limit; a wait
// that runs out records CAOTE_ERR_TIMEOUT and the thread carries on with whatever is in its buffers
// (all indices stay in bounds), so that no thread is left behind at a barrier.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace caote {
namespace prefill {

constexpr int kTile = 128;                  // rows / keys per tile
constexpr int kHalfBytes = kTile * 128;     // one 64-channel box of 128 rows: 16 KB
template <int D>
constexpr int kTileBytesOf = (D / 64) * kHalfBytes;  // a tile of 128 rows
constexpr int kThreads = 128;
constexpr long long kWaitCycles = 2000000000LL;

struct Scratch {
  float* stats;  // [units][Mpad]: minus (log2-domain softmax reference + log2(sum of 2^(s - ref))): alpha = 2^(s + stats)
  float* sstat;  // [units][kTile] LAST_QUERY: the counted rows' statistics side by side (else null)
  float* crest;  // [units][kTile] few: share of all tokens but the counted row's top one (else null)
  float* xpart;  // [units][row blocks][nsplit][D] per CTA of the attention pass: the sum of its counted output rows
  float* ypart;  // [units][cap / sum_keys][D + 4] sum_j base_j v_j over sum_keys keys, at [D] sum_j base_j (else null)
  int* dom;      // [units][2] the slot of the token that holds most of the weight, -1: none, and its h_j
  int sum_keys;  // keys per CTA of carried_sum_kernel
  int Mpad;      // M rounded up to a multiple of kTile
  int nsplit;    // most key splits of the attention pass (1: none)
  int ns;        // key splits of this launch, at most nsplit
  int Ms;        // counted rows per unit
  bool few;      // 0 < Ms < kFewRows: complements without cancellation (see the file comment)
};
constexpr int kFewRows = 64;
// Keys per CTA of carried_sum_kernel: 512, or more where that would be more CTAs (and parts kept in the scratch) than it takes
// to fill the machine many times over: 512 units of 40 000 slots, 21 MB of parts -> 3.
inline int carried_sum_keys(const Dims& dm) {
  int keys = 512;
  while ((long long)dm.units * ((dm.cap + keys - 1) / keys) > 8192 && keys < dm.cap) keys *= 2;
  return keys;
}

// Few units and few query rows leave most SMs idle: the keys of a unit are then cut into up to 8 splits
// that run as the CTAs of a cluster. A function of the shape only.
inline int attn_splits(const Dims& dm) {
  const long long ctas = (long long)((dm.R + kTile - 1) / kTile) * dm.units;
  long long ns = g_sm_count / (ctas > 0 ? ctas : 1);
  const long long max_by_len = ((dm.cap + kTile - 1) / kTile) / 4;  // at least four tiles per split
  if (ns > max_by_len) ns = max_by_len;
  if (ns > 8) ns = 8;
  return ns < 1 ? 1 : (int)ns;
}
// Split plan for a unit of n keys, the last m of them new (device and host agree on it): `ts` tiles per
// split, `count` splits in use. The new block must lie inside the last split, so that every row sees at
// least one key in every split it takes part in.
__host__ __device__ inline void split_plan(int n, int m, int nsplit, int& ts, int& count) {
  const int ntiles = (n + kTile - 1) / kTile;
  for (int k = nsplit; k >= 1; --k) {
    ts = (ntiles + k - 1) / k;
    count = (ntiles + ts - 1) / ts;
    if ((count - 1) * ts * kTile <= n - m) return;
  }
  ts = ntiles;
  count = 1;
}

inline size_t carve(const Dims& dm, char* base, Scratch* out) {
  Scratch s;
  s.Mpad = (dm.R + kTile - 1) / kTile * kTile;
  s.nsplit = attn_splits(dm);
  s.Ms = dm.base_mode == CAOTE_BASE_LAST_QUERY ? dm.G : (dm.base_mode == CAOTE_BASE_EXTERNAL ? 0 : dm.R);
  s.few = s.Ms > 0 && s.Ms < kFewRows;
  s.sum_keys = carried_sum_keys(dm);
  size_t off = 0;
  auto take = [&](bool wanted, size_t n_floats) {
    if (!wanted) return static_cast<float*>(nullptr);
    float* p = reinterpret_cast<float*>(base + off);
    off = align_up(off + sizeof(float) * n_floats, 256);
    return p;
  };
  const size_t units = (size_t)dm.units;
  s.stats = take(true, units * s.Mpad);  // (first: caote_post_evict_output_ws finds it right behind the header)
  s.sstat = take(dm.base_mode == CAOTE_BASE_LAST_QUERY, units * kTile);
  s.crest = take(s.few, units * kTile);
  s.xpart = take(true, units * (s.Mpad / kTile) * s.nsplit * dm.D);
  s.ypart = take(dm.base_mode == CAOTE_BASE_ACCUM || dm.base_mode == CAOTE_BASE_EXTERNAL,
                 units * ((dm.cap + s.sum_keys - 1) / s.sum_keys) * (dm.D + 4));
  s.dom = reinterpret_cast<int*>(take(true, units * 2));
  s.ns = s.nsplit;
  if (out) *out = s;
  return off;
}
// Is row R of a unit one of the rows whose attention defines the base score, and which counted row is it?
__device__ __forceinline__ bool row_counted(const Dims& dm, int R) {
  if (dm.base_mode == CAOTE_BASE_LAST_QUERY) return R % dm.m == dm.m - 1;
  return dm.base_mode != CAOTE_BASE_EXTERNAL;
}
__device__ __forceinline__ int counted_index(const Dims& dm, int R) {
  return dm.base_mode == CAOTE_BASE_LAST_QUERY ? R / dm.m : R;
}

// ---- PTX wrappers (ptx.cuh), the waits built on them, and the tcgen05 wrappers ----------------------------
using ptx::smem_u32;
using ptx::mbar_init;
using ptx::mbar_expect_tx;
using ptx::mbar_arrive;
using ptx::mbar_try_wait;
using ptx::tma_load_2d;
using ptx::bulk_load;
using ptx::fence_async_smem;
using ptx::fast_exp2;
using ptx::tile_off;
// Bounded wait. On expiry the error is recorded and the caller carries on (see the file comment).
__device__ __forceinline__ void mbar_wait(uint64_t* bar, uint32_t parity, int* status) {
  if (mbar_try_wait(bar, parity)) return;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kWaitCycles) {
      set_status(status, CAOTE_ERR_TIMEOUT);
      return;
    }
  }
}
// The same for the single-lane helper warps: they back off between polls so that their spinning does
// not take issue slots from the warps that do the arithmetic on the same scheduler.
__device__ __forceinline__ void mbar_wait_idle(uint64_t* bar, uint32_t parity, int* status) {
  if (mbar_try_wait(bar, parity)) return;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    __nanosleep(20);
    if (clock64() - t0 > kWaitCycles) {
      set_status(status, CAOTE_ERR_TIMEOUT);
      return;
    }
  }
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// TMEM: `cols` columns (a power of two >= 32) for this CTA; one warp allocates, the same warp frees.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_in_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_in_smem)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// Shared-memory matrix descriptor (bf16 tiles staged as 128-byte rows with the 128-byte swizzle).
//   bits [0,14)  start address >> 4        bits [16,30) leading byte offset >> 4
//   bits [32,46) stride byte offset >> 4   bits [46,48) descriptor version (1 on sm_100)
//   bits [61,64) layout type (2 = 128-byte swizzle)
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
// Instruction descriptor of tcgen05.mma.kind::f16: bf16 x bf16 -> fp32, M = 128, N = 128.
//   bits [4,6) D format (1 = f32), [7,10) A format (1 = bf16), [10,13) B format (1 = bf16),
//   bit 15 A major, bit 16 B major (0 = K-major, 1 = MN-major), [17,23) N >> 3, [24,29) M >> 4.
__host__ __device__ constexpr uint32_t instr_desc(bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]; issued by one thread.
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
// The mbarrier gets one arrival once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 32 consecutive fp32 columns of this thread's TMEM lane (lane = 32 * (warp % 4) + lane id).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 64 consecutive columns: half a row of S.
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
      "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
      "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
        "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
        "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
        "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31]),
        "=f"(v[32]), "=f"(v[33]), "=f"(v[34]), "=f"(v[35]), "=f"(v[36]), "=f"(v[37]), "=f"(v[38]), "=f"(v[39]),
        "=f"(v[40]), "=f"(v[41]), "=f"(v[42]), "=f"(v[43]), "=f"(v[44]), "=f"(v[45]), "=f"(v[46]), "=f"(v[47]),
        "=f"(v[48]), "=f"(v[49]), "=f"(v[50]), "=f"(v[51]), "=f"(v[52]), "=f"(v[53]), "=f"(v[54]), "=f"(v[55]),
        "=f"(v[56]), "=f"(v[57]), "=f"(v[58]), "=f"(v[59]), "=f"(v[60]), "=f"(v[61]), "=f"(v[62]), "=f"(v[63])
      : "r"(taddr) : "memory");
}
// The same load of 16 columns without the wait, and the wait as a statement that the registers pass through: whatever reads
// them afterwards depends on the wait, so the compiler cannot move such a read in front of it. Between the two
// the thread may do anything that does not touch r.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
        "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
      :: "memory");
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// Sixteen floats from shared memory, issued where the statement stands (the compiler may not sink it towards the
// first use: the point is to have the loads in flight while other work is done).
__device__ __forceinline__ void lds16_issue(const float* p, float4 (&s)[4]) {
  const uint32_t a = smem_u32(p);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(s[k].x), "=f"(s[k].y), "=f"(s[k].z), "=f"(s[k].w) : "r"(a + 16 * k));
}
__device__ __forceinline__ void tmem_st32u(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]),
        "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),
        "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]: the A operand (K-major, two bf16 per 32-bit column) comes from TMEM.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float x0, float x1) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
  return r;
}
// What k-step ks (16 of the 128 contraction elements) adds to the descriptor of a staged tile.
//   K-major (leading byte offset 16): contraction along the 128-byte rows: 32 bytes per step inside a box, second box after 4.
//   MN-major (leading byte offset kHalfBytes): contraction along the rows of the tile (16 rows = 2 groups of 8 = 2048 bytes per
//   step); the two 64-element boxes along MN are kHalfBytes apart.
__device__ __forceinline__ uint64_t k_major_step(int ks) { return (uint64_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4); }
__device__ __forceinline__ uint64_t mn_major_step(int ks) { return (uint64_t)(ks * 2048 >> 4); }


// ---- attention pass ---------------------------------------------------------------------------------
// Keys are walked in tiles of 128: three K stages, two V stages and the Q block in shared memory, two S buffers,
// and O in TMEM, P (bf16 hi and lo parts) written over the S it came from; the tensor pipe then always has the next
// S = Q K^T queued while the threads are busy with the softmax of the current tile:
//   tensor pipe:  QK(t+1)  PV(t)  QK(t+2)  PV(t+1) ...
//   threads:      softmax(t) ............ softmax(t+1) ...
constexpr int kKeys = 128;                   // keys per tile of the attention pass
constexpr int kKvHalf = kKeys * 128;         // one 64-channel box of 128 keys: 16 KB
constexpr int kKStages = 3;                  // a K stage is free as soon as S is formed
constexpr int kVStages = 2;
constexpr int kRowThreads = 2 * kThreads;    // two threads per query row: each owns 64 of the tile's 128 keys
constexpr int kAttnThreads = kRowThreads + 96;  // + MMA, K-load and V-load warps

// The tensor pipe adds to an fp32 accumulator without rounding to nearest: every addition loses about 2^-25 of the running
// value, always towards zero, so o drifts with the length of the chain (2 x 8 products per tile: 3e-8 x n / 8). After
// every kShare tiles the row threads therefore move O to a second accumulator, which they add to in fp32.
// (n 16 896: error of o against 64 bits 6.5e-5 -> 4.7e-6, what is left is the 16 bits of P; the attention pass 3.03 ->
// 3.01 ms: it is a wait for a product that has nearly finished, and 64 columns, every eighth tile.)
constexpr int kShare = 8;
constexpr int kXchFloats = 7 * kRowThreads;     // half-row maxima and sums in turn, the few-rows form's three closing values, column sums

// Where the splits' rows meet: [split][row of the owner][pitch] floats in the K stages.
template <int D>
constexpr int kMergePitch = D + 4;
static_assert((kTile + 7) * kMergePitch<128> * 4 <= kKStages * kTileBytesOf<128> && (kTile + 7) * kMergePitch<64> * 4 <= kKStages * kTileBytesOf<64>, "");

template <int D>
inline size_t attn_smem_bytes() {
  return 1024 + (size_t)(1 + kKStages + kVStages) * kTileBytesOf<D> + kXchFloats * sizeof(float) + 256;
}

__host__ __device__ constexpr uint32_t instr_desc_n(bool b_mn_major, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// o, row statistics and counted sums of 128 query rows of one unit. grid = (row blocks, units, splits), in clusters of all
// splits of a row block; 352 threads: warps 0..7 are the row threads (two per row); one lane each of warps 8, 9, 10 issues
// the products, the K copies and the V copies.
// tmK / tmV: tensor maps of K and V with boxes of 64 channels x kKeys rows. kFew: the counted rows' largest numerators
// are kept apart (see the file comment).
template <int D, bool kFew>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
            const __grid_constant__ CUtensorMap tmV, Dims dm, const int* __restrict__ len, Scratch sc,
            float* __restrict__ o, int* status) {
  constexpr int kTB = kTileBytesOf<D>, kBoxes = D / 64, kSteps = D / 16;  // k-steps of the first product
  ptx::pdl_wait();
  ptx::pdl_trigger();  // (never before the wait: carried_sum_kernel starts on it and reads what the wait is for)
  extern __shared__ char smem_raw[];
  // (aligned by an offset into the array, not through an integer: the pointer keeps its address space, and what is
  // read and written through it compiles to shared-memory accesses, not generic ones)
  char* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  char* Qs = sm;
  char* Ksm = Qs + kTB;                    // [kKStages]
  char* Vsm = Ksm + kKStages * kTB;        // [kVStages]
  float* xch = reinterpret_cast<float*>(Vsm + kVStages * kTB);  // [kXchFloats]
  uint64_t* bars = reinterpret_cast<uint64_t*>(xch + kXchFloats);
  uint64_t *q_bar = &bars[0], *k_bar = &bars[1], *v_bar = k_bar + kKStages, *s_bar = v_bar + kVStages, *o_bar = s_bar + 2,
           *p_bar = o_bar + 2, *k_free = p_bar + 4, *v_free = k_free + kKStages;  // p_bar: [part][tile parity]
  constexpr int kBars = 1 + 2 * (kKStages + kVStages) + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);

  const int tid = threadIdx.x, lane = tid & 31, warp = ptx::warp_index();
  const int unit = blockIdx.y, row0 = blockIdx.x * kTile;
  const int b = unit / dm.Hkv;
  const int n = len[b], M = dm.R, m = dm.m;
  if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) status[kStatTagIndex] = kStatPerRow;
  if (n == 0) return;  // (the same in the whole cluster)
  if (n < m || n > dm.cap) {
    if (tid == 0) set_status(status, CAOTE_ERR_BAD_LENGTH);
    return;
  }
  // this CTA's share of the unit's key tiles: [kt0, kt0 + ntiles)
  int ts, nsp;
  split_plan(n, m, sc.ns, ts, nsp);
  const int split = blockIdx.z;  // (the rank in the cluster)
  if (split >= nsp) {
    if (nsp > 1) {  // (a unit that runs unsplit has nothing to merge)
      ptx::cluster_sync_all();
      ptx::cluster_sync_all();
    }
    return;
  }
  if (tid == 0 && split == 0 && blockIdx.x == 0) sc.dom[2 * unit] = -1;
  const int kt0 = split * ts;
  const int ntiles = min(ts, (n + kKeys - 1) / kKeys - kt0);
  float* xpart = sc.xpart + ((size_t)unit * gridDim.x * sc.nsplit + blockIdx.x * sc.nsplit + split) * D;

  if (tid == 0) {
    for (int i = 0; i < kBars; ++i) mbar_init(&bars[i], 1);
    for (int i = 0; i < 4; ++i) mbar_init(&p_bar[i], kRowThreads / 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // columns: S0 [0,128), S1 [128,256), O [256,384), the finished shares of O [384,512). P of a tile takes the place of its S once the row threads have
  // read that: hi part in the buffer's columns [0,64), lo part in [64,128) (two bf16 per column), so P is double-
  // buffered like S and the softmax of a tile does not wait for the previous tile's O += P V
  const uint32_t tmem = *tmem_slot;

  if (warp == 9) {
    // =============================== K loads (one lane) ===============================
    if (ptx::elect_one()) {
      mbar_expect_tx(q_bar, kTB);
#pragma unroll
      for (int x = 0; x < kBoxes; ++x) tma_load_2d(Qs + x * kHalfBytes, &tmQ, 64 * x, unit * M + row0, q_bar);
      for (int kt = 0; kt < ntiles; ++kt) {
        const int st = kt % kKStages, row = unit * dm.cap + (kt0 + kt) * kKeys;
        if (kt >= kKStages) mbar_wait_idle(&k_free[st], ((kt / kKStages) - 1) & 1, status);  // S of tile kt - 3 is formed
        mbar_expect_tx(&k_bar[st], kTB);
#pragma unroll
        for (int x = 0; x < kBoxes; ++x) tma_load_2d(Ksm + st * kTB + x * kKvHalf, &tmK, 64 * x, row, &k_bar[st]);
      }
    }
  } else if (warp == 10) {
    // =============================== V loads (one lane) ===============================
    if (ptx::elect_one()) {
      for (int kt = 0; kt < ntiles; ++kt) {
        const int st = kt % kVStages, row = unit * dm.cap + (kt0 + kt) * kKeys;
        if (kt >= kVStages) mbar_wait_idle(&v_free[st], ((kt / kVStages) - 1) & 1, status);  // O += P V of tile kt - 2 is done
        mbar_expect_tx(&v_bar[st], kTB);
#pragma unroll
        for (int x = 0; x < kBoxes; ++x) tma_load_2d(Vsm + st * kTB + x * kKvHalf, &tmV, 64 * x, row, &v_bar[st]);
      }
    }
  } else if (warp == 8) {
    // =============================== products (one lane) ===============================
    if (ptx::elect_one()) {
      constexpr uint32_t kIdescS = instr_desc_n(false, kKeys), kIdescO = instr_desc_n(true, D);
      const uint32_t q_addr = smem_u32(Qs);
      const uint64_t qdesc0 = smem_desc(q_addr, 16, 1024);
      const uint64_t kdesc0 = smem_desc(smem_u32(Ksm), 16, 1024);
      const uint64_t vdesc0 = smem_desc(smem_u32(Vsm), kKvHalf, 1024);
      auto issue_qk = [&](int kt) {
        mbar_wait(&k_bar[kt % kKStages], (kt / kKStages) & 1, status);
        tc_fence_after();
        const uint64_t kd = kdesc0 + (uint64_t)(((kt % kKStages) * kTB) >> 4);
        const uint32_t d_s = tmem + (kt & 1) * kKeys;  // S0 or S1
#pragma unroll
        for (int ks = 0; ks < kSteps; ++ks) umma(d_s, qdesc0 + k_major_step(ks), kd + k_major_step(ks), kIdescS, ks > 0);
        umma_commit(&s_bar[kt & 1]);
        umma_commit(&k_free[kt % kKStages]);
      };
      mbar_wait(q_bar, 0, status);
      issue_qk(0);
      for (int kt = 0; kt < ntiles; ++kt) {
        // queue S of the next tile: its buffer was read by the softmax of tile kt - 1, which has
        // arrived on p_bar before PV(kt - 1) was issued
        if (kt + 1 < ntiles) issue_qk(kt + 1);
        // O += P V as the rows write P of this tile: the first 32 keys of either half, then the others
        mbar_wait(&v_bar[kt % kVStages], (kt / kVStages) & 1, status);
        const uint64_t vd = vdesc0 + (uint64_t)(((kt % kVStages) * kTB) >> 4);
        const uint32_t p_tmem = tmem + (kt & 1) * kKeys;
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          mbar_wait(&p_bar[2 * part + (kt & 1)], (kt >> 1) & 1, status);
          tc_fence_after();
#pragma unroll
          for (int i = 0; i < 4; ++i) {  // 16 keys = 8 packed columns per step
            const int ks = (i >> 1) * 4 + 2 * part + (i & 1);
            umma_ts(tmem + 256, p_tmem + ks * 8, vd + mn_major_step(ks), kIdescO, ks > 0 || kt % kShare > 0);  // (a new share starts at 0)
            umma_ts(tmem + 256, p_tmem + 64 + ks * 8, vd + mn_major_step(ks), kIdescO, true);
          }
        }
        umma_commit(&o_bar[kt & 1]);
        umma_commit(&v_free[kt % kVStages]);
      }
    }
  } else {
    // =============================== two threads per query row ===============================
    // Thread t and thread t + 128 share row t of the block: each owns 64 of a tile's 128 keys (and 64
    // of the 128 output channels when O is rescaled or written out). They agree on the softmax
    // reference through a two-float exchange in shared memory and a barrier of the two warps that share the rows.
    const int rowl = tid & (kThreads - 1), half = tid >> 7;
    const int R = row0 + rowl;
    const int nvis = (R < M) ? n - m + (R % m) + 1 : n;  // keys this row sees (causal inside the block)
    const float scale2 = dm.scale * 1.4426950408889634f;
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_o = t_lane + 256 + half * (D / 2);
    float m_ref = -INFINITY, l = 0.f;
    // few counted rows (kFew): this thread's largest product, its numerator and the sum of the other numerators; warps
    // without a counted row skip that (summing the exponentials a second time instead: 158 us against 104 us at 16 units,
    // 896 rows, 6 128 tokens)
    float smax = -INFINITY, ptop = 0.f, lrest = 0.f;
    const bool counted = kFew && R < M && row_counted(dm, R);
    const bool keep_top = kFew && __any_sync(0xffffffffu, counted);

    if (ntiles > kShare) {  // the sum of finished shares starts at 0
      const uint32_t zero[16] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int cc = 0; cc < D / 32; ++cc) tmem_st16u(t_o + 128 + cc * 16, zero);
      tmem_st_wait();
    }
    for (int kt = 0; kt < ntiles; ++kt) {
      mbar_wait(&s_bar[kt & 1], (kt >> 1) & 1, status);
      tc_fence_after();
      const int j0 = (kt0 + kt) * kKeys + half * 64;  // first key of this thread's half
      const uint32_t t_s = t_lane + (kt & 1) * kKeys + half * 64;
      float sv[64];  // raw products; masked keys become -inf
      tmem_ld64(t_s, sv);
      if ((kt0 + kt) * kKeys + kKeys > n - m + 1) {  // only tiles that reach into the new block (or past the length) need the mask
#pragma unroll
        for (int i = 0; i < 64; ++i) sv[i] = (j0 + i < nvis) ? sv[i] : -INFINITY;
      }
      float raw_top;  // (scale2 > 0: the largest product is the largest logit)
      {
        float pm[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pm[i] = fmaxf(sv[i], sv[i + 8]);
#pragma unroll
        for (int i = 16; i < 64; i += 16) {
#pragma unroll
          for (int e = 0; e < 8; ++e) pm[e] = fmaxf(fmaxf(pm[e], sv[i + e]), sv[i + 8 + e]);
        }
        raw_top = fmaxf(fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3])), fmaxf(fmaxf(pm[4], pm[5]), fmaxf(pm[6], pm[7])));
      }
      float mx = raw_top * scale2;
      // the other half of the row (the two warps that share 32 rows meet here; each writes P over columns of S that the other has
      // read, hence the fences)
      float* xm = xch + (kt & 1) * kRowThreads;
      xm[tid] = mx;
      tc_fence_before();
      asm volatile("bar.sync %0, 64;" ::"r"(2 + (warp & 3)) : "memory");
      tc_fence_after();
      mx = fmaxf(mx, xm[tid ^ kThreads]);
      // the reference moves only when a logit exceeds it by more than 8 (p <= 256 in between)
      const bool need = mx > m_ref + 8.f;
      const bool close = kt > 0 && kt % kShare == 0;  // O holds a finished share
      float corr = 1.f;
      if (need) {
        corr = fast_exp2(m_ref - mx);
        m_ref = mx;
        l *= corr;
        if (kFew) { ptop *= corr; lrest *= corr; }
      }
      const float2 scale22 = make_float2(scale2, scale2), neg_ref2 = make_float2(-m_ref, -m_ref);
      float2 ls[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      float rs[2] = {0.f, 0.f};
      // P goes where S was: both halves of the row have read their S columns (the barrier above), and the
      // product that read the buffer's previous P was issued before the product that formed this S
      const uint32_t t_p = t_lane + (kt & 1) * kKeys + half * 32;  // this half's 64 keys = 32 packed columns
      // 32 of the half's keys at a time, so that the product over the first part runs while the second is formed
      auto numerators = [&](int part, auto top) {  // top: rs sums the numerators of all keys but the tile's largest
        uint32_t hi[16], lo[16];  // column c = keys 2c (low half) and 2c + 1
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          // P = hi + lo, hi truncated and lo rounded to bf16 (16 significant bits together); plain bit
          // operations, so the conversion unit is left to the exponentials
          const int i = 32 * part + 2 * c;
          const float2 e = __ffma2_rn(make_float2(sv[i], sv[i + 1]), scale22, neg_ref2);
          const float2 p = make_float2(fast_exp2(e.x), fast_exp2(e.y));
          const uint32_t b0 = __float_as_uint(p.x), b1 = __float_as_uint(p.y);
          hi[c] = __byte_perm(b0, b1, 0x7632);
          const float2 r = __ffma2_rn(make_float2(__uint_as_float(b0 & 0xffff0000u), __uint_as_float(b1 & 0xffff0000u)),
                                      make_float2(-1.f, -1.f), p);
          lo[c] = __byte_perm(__float_as_uint(r.x) + 0x8000u, __float_as_uint(r.y) + 0x8000u, 0x7632);  // rounded
          ls[c & 1] = __fadd2_rn(ls[c & 1], p);
          if constexpr (decltype(top)::value) {
            if (sv[i] != raw_top) rs[c & 1] += p.x;
            if (sv[i + 1] != raw_top) rs[c & 1] += p.y;
          }
        }
        tmem_st16u(t_p + 16 * part, hi);
        tmem_st16u(t_p + 64 + 16 * part, lo);
      };
      auto form = [&](int part) {
        if (kFew && keep_top) numerators(part, std::true_type{});
        else numerators(part, std::false_type{});
      };
      form(0);
      // O += P V of the previous tile has finished by now, or nearly: O is rescaled, a finished share moved, before the first
      // product of this tile is queued
      if (kt > 0 && (close || __any_sync(0xffffffffu, need))) {
        mbar_wait(&o_bar[(kt - 1) & 1], ((kt - 1) >> 1) & 1, status);
        tc_fence_after();
        // (rolled loops: this code is seldom run, and has to be fetched every time)
        if (close) {
#pragma unroll 1
          for (int cc = 0; cc < D / 32; ++cc) {
            uint32_t v[16], w[16];
            tmem_ld16_issue(t_o + cc * 16, v);
            tmem_ld16_issue(t_o + 128 + cc * 16, w);
            tmem_ld16_wait(v);
            tmem_ld16_wait(w);
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = __float_as_uint((__uint_as_float(v[i]) + __uint_as_float(w[i])) * corr);
            tmem_st16u(t_o + 128 + cc * 16, w);
          }
        } else {
#pragma unroll 1
          for (int cc = 0; cc < (kt > kShare ? D / 16 : D / 32); ++cc) {  // O, and the sum of earlier shares if there is one
            const uint32_t at = t_o + (cc / (D / 32)) * 128 + (cc % (D / 32)) * 16;
            uint32_t v[16];
            tmem_ld16_issue(at, v);
            tmem_ld16_wait(v);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * corr);
            tmem_st16u(at, v);
          }
        }
      }
      const int n_valid = min(kKeys, n - (kt0 + kt) * kKeys);
      if (n_valid < kKeys) {
        // V rows behind the unit's length: clear them so that 0 * (stray NaN) cannot reach O
        mbar_wait(&v_bar[kt % kVStages], (kt / kVStages) & 1, status);
        if (tid < kKeys && tid >= n_valid) {
          char* vt = Vsm + (kt % kVStages) * kTB;
#pragma unroll
          for (int c = 0; c < D / 8; ++c)
            *reinterpret_cast<uint4*>(vt + (c >> 3) * kKvHalf + tid * 128 + (((c & 7) ^ (tid & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_async_smem();
      }
      auto hand_over = [&](int part) {
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_bar[2 * part + (kt & 1)]);
      };
      hand_over(0);
      form(1);
      hand_over(1);
      const float lt = (ls[0].x + ls[0].y) + (ls[1].x + ls[1].y);
      l += lt;
      if (kFew && keep_top) {
        // one copy of the tile's largest numerator stays apart, any other copies join the rest (their number from the
        // two sums: pt is the largest of 64 terms, so the sums' rounding is far below half of it)
        const float pt = fast_exp2(fmaf(raw_top, scale2, -m_ref)), rt = rs[0] + rs[1];
        float r = rt + (pt > 0.f ? rintf((lt - rt) / pt) - 1.f : 0.f) * pt;
        const bool bigger = raw_top > smax;
        r += bigger ? ptop : pt;
        lrest += r;
        ptop = bigger ? pt : ptop;
        smax = bigger ? raw_top : smax;
      }
    }
    mbar_wait(&o_bar[(ntiles - 1) & 1], ((ntiles - 1) >> 1) & 1, status);
    tc_fence_after();

    // ---- normalise and write out: the two halves of a row add up their sums first ----
    float* xl = xch + (ntiles & 1) * kRowThreads;  // the copy the last tile did not use
    xl[tid] = l;
    asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
    l += xl[tid ^ kThreads];
    if (kFew) {
      // the two halves' (sum of the others, largest numerator, its logit): the larger one stays apart
      float* xt = xch + 2 * kRowThreads;
      xt[tid] = lrest;
      xt[kRowThreads + tid] = ptop;
      xt[2 * kRowThreads + tid] = smax;
      asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
      const int other = tid ^ kThreads;
      const float op = xt[kRowThreads + other], os = xt[2 * kRowThreads + other];
      const bool keep = smax > os || (smax == os && half == 0);
      lrest += xt[other] + (keep ? op : ptop);
      ptop = keep ? ptop : op;
      smax = fmaxf(smax, os);
    }
    // this split's output, normalised by its own sum, and its statistics
    const float inv_l = 1.f / l;
    float ov[D / 64][32];
#pragma unroll
    for (int cc = 0; cc < D / 64; ++cc) {
      tmem_ld32(t_o + cc * 32, ov[cc]);
      if (ntiles > kShare) {
        float w[32];
        tmem_ld32(t_o + 128 + cc * 32, w);
#pragma unroll
        for (int i = 0; i < 32; ++i) ov[cc][i] += w[i];
      }
    }
    const bool in_x = R < M && row_counted(dm, R);
    if (nsp == 1) {
      // straight out; the column sums of the counted rows by halving: after the step over lanes 16 apart a lane keeps half
      // of its channels, and so on; in the end lane l of a warp holds D / 64 channels of its 32 rows
#pragma unroll
      for (int cc = 0; cc < D / 64; ++cc) {
        float* orow = o + ((size_t)unit * M + R) * D + half * (D / 2) + cc * 32;
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 v = make_float4(ov[cc][i] * inv_l, ov[cc][i + 1] * inv_l, ov[cc][i + 2] * inv_l, ov[cc][i + 3] * inv_l);
          if (R < M) *reinterpret_cast<float4*>(orow + i) = v;
          ov[cc][i] = in_x ? v.x : 0.f; ov[cc][i + 1] = in_x ? v.y : 0.f; ov[cc][i + 2] = in_x ? v.z : 0.f; ov[cc][i + 3] = in_x ? v.w : 0.f;
        }
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
          const bool up = (tid & w) != 0;
#pragma unroll
          for (int i = 0; i < w; ++i) {
            const float send = up ? ov[cc][i] : ov[cc][i + w], keep = up ? ov[cc][i + w] : ov[cc][i];
            ov[cc][i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
          }
        }
        xch[5 * kRowThreads + (warp & 3) * D + half * (D / 2) + cc * 32 + (tid & 31)] = ov[cc][0];  // (lane l has channel l)
      }
      if (R < M && half == 0) {
        const float stat = -(m_ref + __log2f(l));
        sc.stats[(size_t)unit * sc.Mpad + R] = stat;
        if (kFew && in_x) {
          if (sc.sstat) sc.sstat[(size_t)unit * kTile + counted_index(dm, R)] = stat;
          sc.crest[(size_t)unit * kTile + counted_index(dm, R)] = lrest / (lrest + ptop);
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
      if (tid < D) {
        const float* part = xch + 5 * kRowThreads + tid;
        xpart[tid] = (part[0] + part[D]) + (part[2 * D] + part[3 * D]);
      }
    } else {
      // ... go to the CTA of the cluster that owns the row (its K stages; the row pitch keeps the lanes of a store on
      // different banks), once that one is through with its tiles
      const int rp = (kTile + nsp - 1) / nsp, owner = rowl / rp, rl = rowl - owner * rp;
      __syncwarp();
      ptx::cluster_sync_all();
      const uint32_t dst = ptx::map_to_rank(smem_u32(Ksm) + (uint32_t)(((split * rp + rl) * kMergePitch<D> + half * (D / 2)) * 4), owner);
#pragma unroll
      for (int cc = 0; cc < D / 64; ++cc)
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          ptx::st_dsmem_v4(dst + (cc * 32 + i) * 4, make_uint4(__float_as_uint(ov[cc][i] * inv_l), __float_as_uint(ov[cc][i + 1] * inv_l),
                                                               __float_as_uint(ov[cc][i + 2] * inv_l), __float_as_uint(ov[cc][i + 3] * inv_l)));
      if (half == 0)
        ptx::st_dsmem_v4(ptx::map_to_rank(smem_u32(xch) + (uint32_t)((split * rp + rl) * 16), owner),
                         make_uint4(__float_as_uint(m_ref + __log2f(l)), __float_as_uint(smax), __float_as_uint(kFew ? lrest / (lrest + ptop) : 0.f), 0u));
    }
  }
  if (nsp > 1) {
    __syncwarp();
    if (warp >= 8) ptx::cluster_sync_all();
    ptx::cluster_sync_all();  // every split's rows have arrived; from here on the CTA reads its own shared memory only
  }

  if (nsp > 1 && warp < 8) {
    // ---- merge: o = sum_s o_s 2^(stat_s - stat), stat = log2 sum_s 2^stat_s; a warp per row, lane = D / 32 channels ----
    constexpr int CPL = D / 32;
    const int rp = (kTile + nsp - 1) / nsp;
    const float4* rst = reinterpret_cast<const float4*>(xch);  // [split][row]: statistic, largest product, the others' share
    float cs[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) cs[c] = 0.f;
    for (int rl = warp; rl < rp; rl += 8) {
      const int R = row0 + split * rp + rl;
      if (split * rp + rl >= kTile || R >= M) break;
      float mx = -INFINITY, tot = 0.f, acc[CPL], wgt[8];
#pragma unroll
      for (int c = 0; c < CPL; ++c) acc[c] = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        wgt[u] = u < nsp ? rst[u * rp + rl].x : -INFINITY;
        mx = fmaxf(mx, wgt[u]);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (u < nsp) {
          wgt[u] = fast_exp2(wgt[u] - mx);
          tot += wgt[u];
          const float* p = reinterpret_cast<const float*>(Ksm) + (u * rp + rl) * kMergePitch<D> + lane * CPL;
          if constexpr (CPL == 4) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            acc[0] = fmaf(v.x, wgt[u], acc[0]); acc[1] = fmaf(v.y, wgt[u], acc[1]);
            acc[2] = fmaf(v.z, wgt[u], acc[2]); acc[3] = fmaf(v.w, wgt[u], acc[3]);
          } else {
            const float2 v = *reinterpret_cast<const float2*>(p);
            acc[0] = fmaf(v.x, wgt[u], acc[0]); acc[1] = fmaf(v.y, wgt[u], acc[1]);
          }
        }
      }
      const float inv = 1.f / tot;
      const bool in_x = row_counted(dm, R);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        acc[c] *= inv;
        if (in_x) cs[c] += acc[c];
      }
      float* orow = o + ((size_t)unit * M + R) * D + lane * CPL;
      if constexpr (CPL == 4) *reinterpret_cast<float4*>(orow) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      else *reinterpret_cast<float2*>(orow) = make_float2(acc[0], acc[1]);
      if (lane == 0) {
        const float stat = -(mx + __log2f(tot));
        sc.stats[(size_t)unit * sc.Mpad + R] = stat;
        if (kFew && in_x) {
          const int q = counted_index(dm, R);
          if (sc.sstat) sc.sstat[(size_t)unit * kTile + q] = stat;
          // all tokens but the row's top one: the other splits, and the rest of the split that holds it
          float top = -INFINITY, rest = 0.f;
          int at = 0;
          for (int u = 0; u < nsp; ++u) {
            const float v = rst[u * rp + rl].y;
            if (v > top) { top = v; at = u; }
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < nsp) rest += wgt[u] * (u == at ? rst[u * rp + rl].z : 1.f);
          sc.crest[(size_t)unit * kTile + q] = rest * inv;
        }
      }
    }
    // the warps' sums, in a fixed order
    float* wcs = reinterpret_cast<float*>(Vsm);
#pragma unroll
    for (int c = 0; c < CPL; ++c) wcs[warp * D + lane * CPL + c] = cs[c];
    asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
    if (tid < D) {
      float x = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) x += wcs[w * D + tid];
      xpart[tid] = x;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Parts of sum_j base_j v_j and sum_j base_j: grid = (ceil(cap / sc.sum_keys), units), 256 threads. A thread takes one 16-byte
// piece of every (256 / pieces)-th row, eight rows in flight; the rows' groups add up in shared memory in a fixed order.
// No wait at the top (32 units of 7.3 k tokens: 23 us in the merge of the splits -> hidden behind the attention pass; a spare
// warp of that kernel adding up the V tiles in shared memory held them too long: attention 102 -> 194 us). That is sound only
// because the launch right before it is attn_kernel's, every CTA of which is past its own wait before it triggers this one:
// all that came before has then completed and written back, the appended rows, the carried scores, and the last reader of
// this scratch. A grid that has not waited for itself is promised no view of that but the one in L2, so lengths, scores and
// rows are read there (ld.global.cg), not through a cache that may have seen them earlier.
template <int D>
__global__ void __launch_bounds__(256)
carried_sum_kernel(Dims dm, const int* len, Scratch sc, const float* base, const __nv_bfloat16* V) {
  constexpr int P = D / 8, kGroups = 256 / P, kFly = 8;
  __shared__ float part[kGroups][D + 1];
  ptx::pdl_trigger();
  const int unit = blockIdx.y, n = __ldcg(len + unit / dm.Hkv), j0 = blockIdx.x * sc.sum_keys;
  const int piece = threadIdx.x % P, g = threadIdx.x / P;
  const bool work = n >= dm.m && n <= dm.cap && j0 < n;
  if (work) {
    const int j1 = min(n, j0 + sc.sum_keys);
    const float* bu = base + (size_t)unit * dm.cap;
    const uint4* src = reinterpret_cast<const uint4*>(V + (size_t)unit * dm.cap * D) + piece;
    float2 y[4];
    float hb = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) y[e] = make_float2(0.f, 0.f);
    for (int j = j0 + g; j < j1; j += kFly * kGroups) {
      float b[kFly];
      uint4 raw[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const bool in = j + u * kGroups < j1;
        b[u] = in ? __ldcg(bu + j + u * kGroups) : 0.f;
        raw[u] = in ? __ldcg(src + (size_t)(j + u * kGroups) * P) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
        hb += b[u];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          y[e] = __ffma2_rn(make_float2(b[u], b[u]), make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)), y[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      part[g][8 * piece + 2 * e] = y[e].x;
      part[g][8 * piece + 2 * e + 1] = y[e].y;
    }
    if (piece == 0) part[g][D] = hb;
  }
  __syncthreads();
  if (work && threadIdx.x <= D) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) t += part[i][threadIdx.x];
    sc.ypart[((size_t)unit * gridDim.x + blockIdx.x) * (D + 4) + threadIdx.x] = t;
  }
  ptx::pdl_wait();  // (whoever waits for this kernel waits for the attention pass with it)
}

// X of a unit from its parts (see the file comment), by one warp: lane = D / 32 channels of x; returns sum_j base_j.
// vsum: FastCAOTE, X is the mean of the cached values.
template <int D>
__device__ __forceinline__ float x_from_parts(const Dims& dm, const Scratch& sc, int unit, int n, const float* __restrict__ vsum,
                                              int lane, float (&x)[D / 32]) {
  constexpr int CPL = D / 32, kFly = 8;
  float hb = 0.f;
#pragma unroll
  for (int c = 0; c < CPL; ++c) x[c] = vsum ? vsum[(size_t)unit * D + lane * CPL + c] : 0.f;
  if (!vsum && sc.Ms > 0) {
    int ts, nsp;
    split_plan(n, dm.m, sc.ns, ts, nsp);
    const int nrb = sc.Mpad / kTile, parts = nrb * nsp;
    const float* xp = sc.xpart + (size_t)unit * nrb * sc.nsplit * D + lane * CPL;
    for (int p0 = 0; p0 < parts; p0 += kFly) {
      float v[kFly][CPL];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const int p = min(p0 + u, parts - 1);
#pragma unroll
        for (int c = 0; c < CPL; ++c) v[u][c] = xp[(size_t)((p / nsp) * sc.nsplit + p % nsp) * D + c];
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u)
        if (p0 + u < parts) {
#pragma unroll
          for (int c = 0; c < CPL; ++c) x[c] += v[u][c];
        }
    }
  }
  if (sc.ypart) {
    const int parts = (n + sc.sum_keys - 1) / sc.sum_keys;
    const float* yp = sc.ypart + (size_t)unit * ((dm.cap + sc.sum_keys - 1) / sc.sum_keys) * (D + 4);
    for (int p0 = 0; p0 < parts; p0 += kFly) {
      float v[kFly][CPL], h[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const float* at = yp + (size_t)min(p0 + u, parts - 1) * (D + 4);
#pragma unroll
        for (int c = 0; c < CPL; ++c) v[u][c] = at[lane * CPL + c];
        h[u] = at[D];
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u)
        if (p0 + u < parts) {
          hb += h[u];
          if (!vsum) {
#pragma unroll
            for (int c = 0; c < CPL; ++c) x[c] += v[u][c];
          }
        }
    }
  }
  const float H = vsum ? (float)n : (float)sc.Ms + hb;
#pragma unroll
  for (int c = 0; c < CPL; ++c) x[c] = H > 0.f ? x[c] / H : 0.f;
  return hb;
}

// Share of a unit's weight above which a token's score is dominant_kernel's. Below it the plain differences are good to about
// 3e-6 / (1 - w), 3e-5 of the score at the line.
constexpr float kDominant = 0.9f;
constexpr int kScoreKeys = 2 * kTile;            // keys per work item: two key tiles share every Q block
constexpr int kKeyThreads = 2 * kScoreKeys;       // two threads per key: each owns 64 of a block's 128 rows
constexpr int kScoreThreads = kKeyThreads + 96;   // + a warp for the products, one for K, V and X, one for Q and the statistics
constexpr int kQStages = 2;                       // Q blocks: a stage is free again once its products are done
constexpr int kSStages = 8;                       // their rows' statistics: free once the key threads have used them
template <bool kFew>
constexpr int kStatFloatsOf = kFew ? 2 * kTile : kTile;  // the statistics of a block's 128 rows (few: and their crest)

template <int D>
inline size_t score_smem_bytes() {
  return 1024 + (4 + kQStages) * (size_t)kTileBytesOf<D> + (kSStages * 2 * kTile + 2 * (D + 4) + 6 * kScoreKeys) * sizeof(float) + 320;
}

// 2^x for two arguments at once on the FMA pipe instead of the special-function unit: x = i + f with i the nearest
// integer (taken from the low bits of x + 1.5 * 2^23), 2^f on [-1/2, 1/2] by a polynomial of degree 4 that is exact at
// f = 0 (relative error below 3e-6), and i added to the exponent field. Arguments below -126 give about 2^-126.
// The score pass is bound by the special-function unit's 16 results per clock and SM (one exponential per
// (row, key) pair); it hands a quarter of them to this routine.
__device__ __forceinline__ float2 poly_exp2x2(float2 x) {
  constexpr float kMagic = 12582912.f;
  x.x = fmaxf(x.x, -126.f);
  x.y = fmaxf(x.y, -126.f);
  const float2 t = __fadd2_rn(x, make_float2(kMagic, kMagic));
  const float2 r = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
  const float2 f = __ffma2_rn(r, make_float2(-1.f, -1.f), x);
  float2 p = __ffma2_rn(make_float2(0.009589649736881256f, 0.009589649736881256f), f,
                        make_float2(0.05590599775314331f, 0.05590599775314331f));
  p = __ffma2_rn(p, f, make_float2(0.24023915827274323f, 0.24023915827274323f));
  p = __ffma2_rn(p, f, make_float2(0.6931241154670715f, 0.6931241154670715f));
  p = __ffma2_rn(p, f, make_float2(1.f, 1.f));
  return make_float2(__int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23)),
                     __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23)));
}

// Adds to a key's running sum the attention weights 2^(s * scale2 + statistic) of 16 rows (v: the logits of the
// key against these rows, st: the rows' statistics). plain: no row is masked. Of every eight exponentials six go to
// the special-function unit and two to the polynomial.
__device__ __forceinline__ void score_piece16(const uint32_t (&v)[16], const float4 (&st)[4], float scale2, bool plain,
                                              int R0, int M, int m, int need, float2 (&hacc)[2], float& hmasked) {
  if (plain) {
    const float2 sc2 = make_float2(scale2, scale2);
    auto arg = [&](int i, float s0, float s1) {
      return __ffma2_rn(make_float2(__uint_as_float(v[i]), __uint_as_float(v[i + 1])), sc2, make_float2(s0, s1));
    };
#pragma unroll
    for (int i = 0; i < 16; i += 8) {
      const float4 ra = st[i / 4], rb = st[i / 4 + 1];
      const float2 e0 = arg(i, ra.x, ra.y), e1 = arg(i + 2, ra.z, ra.w), e2 = arg(i + 4, rb.x, rb.y);
      hacc[0] = __fadd2_rn(hacc[0], make_float2(fast_exp2(e0.x), fast_exp2(e0.y)));
      hacc[1] = __fadd2_rn(hacc[1], make_float2(fast_exp2(e1.x), fast_exp2(e1.y)));
      hacc[0] = __fadd2_rn(hacc[0], make_float2(fast_exp2(e2.x), fast_exp2(e2.y)));
      hacc[1] = __fadd2_rn(hacc[1], poly_exp2x2(arg(i + 6, rb.z, rb.w)));
    }
  } else {
    // row R sees key j iff j <= n - m + (R % m), i.e. iff (R % m) >= need; R % m is carried along instead of
    // being divided out for every pair
    const float stf[16] = {st[0].x, st[0].y, st[0].z, st[0].w, st[1].x, st[1].y, st[1].z, st[1].w,
                           st[2].x, st[2].y, st[2].z, st[2].w, st[3].x, st[3].y, st[3].z, st[3].w};
    int rm = R0 % m;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const bool vis = (R0 + i < M) && (rm >= need);
      const float a = fast_exp2(fmaf(__uint_as_float(v[i]), scale2, stf[i]));
      hmasked += vis ? a : 0.f;
      if (++rm == m) rm = 0;
    }
  }
}

// The same for a few counted rows: besides the weights, the complements 1 - alpha of the key; a weight above one half
// belongs to the row's top token, whose complement the attention pass has left in crest.
__device__ __forceinline__ void score_piece16_few(const uint32_t (&v)[16], const float4 (&st)[4], const float* crest, float scale2,
                                                  int R0, int M, int m, int need, float& h, float& rest) {
  if (R0 >= M) return;
  const float stf[16] = {st[0].x, st[0].y, st[0].z, st[0].w, st[1].x, st[1].y, st[1].z, st[1].w,
                         st[2].x, st[2].y, st[2].z, st[2].w, st[3].x, st[3].y, st[3].z, st[3].w};
  int rm = R0 % m;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const bool row = R0 + i < M;
    const float a = (row && rm >= need) ? fast_exp2(fmaf(__uint_as_float(v[i]), scale2, stf[i])) : 0.f;
    h += a;
    rest += row ? (a > 0.5f ? crest[i] : 1.f - a) : 0.f;
    if (++rm == m) rm = 0;
  }
}

// CAOTE scores, 256 keys of a unit at a time (an item). The grid is one CTA per SM and walks the items with a stride of its
// size, so that an item's K tiles are fetched while the one before it is summed, its value rows while its own last blocks
// are, and the products of the next item start before the scores of this one are written. (A CTA per item: 32 units of 7.3 k
// keys x 512 rows 82 us, of which every CTA spent 4 of 10.5 us on set-up, the first copies and the value rows; now 71.)
// 608 threads: warps 0..15 are the key threads, two per key (warps 0..3 and 8..11 the first key tile, 4..7 and 12..15 the
// second; the lower eight take rows 0..63 of every Q block and the lower half of the channels, the upper eight the others),
// one lane each of warps 16, 17, 18 issues the products, the copies of K and V, and those of Q and the statistics; warp 17
// also adds up X of the item's unit (a warp of its own for that cost 3 % on long blocks of queries).
// Two buffers of two tiles take turns: K of item i, then its V once the last product has read K, then K of item i + 2.
// tmQ: the counted rows (LAST_QUERY: the last row of every head). kFew: complements without cancellation; kAccum: carried
// scores are added and written back.
template <int D, bool kFew, bool kAccum>
__global__ void __launch_bounds__(kScoreThreads, 1)
score_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
             const __grid_constant__ CUtensorMap tmV, Dims dm, const int* __restrict__ len, Scratch sc,
             float* __restrict__ base, float* __restrict__ scores, const float* __restrict__ vsum, int* status) {
  constexpr int kTB = kTileBytesOf<D>, kBoxes = D / 64, kSteps = D / 16, kSF = kStatFloatsOf<kFew>;
  ptx::pdl_wait();
  ptx::pdl_trigger();
  extern __shared__ char smem_raw[];
  // (aligned by an offset into the array, not through an integer: the pointer keeps its address space, and what is
  // read and written through it compiles to shared-memory accesses, not generic ones)
  char* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  char* KVs = sm;                                               // [2][2] tiles: K, later V, of an item
  char* Qst = KVs + 4 * kTB;                                    // [kQStages] Q blocks
  float* Sst = reinterpret_cast<float*>(Qst + kQStages * kTB);  // [kSStages][kSF] row statistics (few: then their crest)
  float* Xs = Sst + kSStages * 2 * kTile;                       // [2][D + 4]; at [D] the sum of the carried scores
  float* hx = Xs + 2 * (D + 4);                                       // [2][kScoreKeys] upper halves' sums,
  float* ax = hx + 2 * kScoreKeys;                              // [2][kScoreKeys] squared distances,
  float* rx = ax + 2 * kScoreKeys;                              // [2][kScoreKeys] few: complements
  uint64_t* bars = reinterpret_cast<uint64_t*>(rx + 2 * kScoreKeys);
  uint64_t *k_full = &bars[0], *k_done = k_full + 2, *v_full = k_done + 2, *q_full = v_full + 2, *q_done = q_full + kQStages,
           *st_full = q_done + kQStages, *s_bar = st_full + kSStages, *v_free = s_bar + 2, *c_bar = v_free + 2, *st_free = c_bar + 2;
  constexpr int kBars1 = 6 + 2 * kQStages + kSStages + 2;  // single arrivals (a copy's bytes, a commit)
  constexpr int kBars = kBars1 + 4 + kSStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);

  const int tid = threadIdx.x, warp = ptx::warp_index();
  const bool last_only = kFew && dm.base_mode == CAOTE_BASE_LAST_QUERY;
  const int M = kFew ? sc.Ms : dm.R, m = last_only ? 1 : dm.m;  // counted rows, and the block they are causal in
  const int nblocks = (M + kTile - 1) / kTile;
  const int per_unit = (dm.cap + kScoreKeys - 1) / kScoreKeys, items = dm.units * per_unit;
  // the next item at or behind `it` that holds keys (its unit, first key and the unit's length); false: no more
  int it = blockIdx.x, unit = 0, j0 = 0, n = 0;
  auto next = [&]() {
    for (; it < items; it += gridDim.x) {
      unit = it / per_unit;
      j0 = (it - unit * per_unit) * kScoreKeys;
      n = __ldg(len + unit / dm.Hkv);
      if (n >= dm.m && n <= dm.cap && j0 < n) {
        it += gridDim.x;
        return true;
      }
    }
    return false;
  };

  if (tid == 0) {
    for (int i = 0; i < kBars1; ++i) mbar_init(&bars[i], 1);
    for (int i = kBars1; i < kBars; ++i) mbar_init(&bars[i], kKeyThreads / 32);  // one arrival per key warp
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;  // key tile kk, buffer buf: columns [kk * 256 + buf * 128, + 128)

  if (warp == 17) {
    // =============================== copies of K and V (one lane), X of the item's unit (the warp) ===============================
    const int lane = tid & 31;
    auto load_pair = [&](int buf, const CUtensorMap* tm, uint64_t* bar, int u, int first) {
      mbar_expect_tx(bar, 2 * kTB);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk)
#pragma unroll
        for (int x = 0; x < kBoxes; ++x)
          tma_load_2d(KVs + (2 * buf + kk) * kTB + x * kHalfBytes, tm, 64 * x, u * dm.cap + first + kk * kTile, bar);
    };
    bool more = next();
    if (more && lane == 0) load_pair(0, &tmK, &k_full[0], unit, j0);
    for (int c = 0; more; ++c) {
      const int buf = c & 1, u = unit, first = j0;
      float x[D / 32];
      const float hb = x_from_parts<D>(dm, sc, unit, n, vsum, lane, x);
      // (K of this item went into buffer `buf` after v_free said that the item before last is done with it, and with its X)
#pragma unroll
      for (int i = 0; i < D / 32; ++i) Xs[buf * (D + 4) + lane * (D / 32) + i] = x[i];
      if (lane == 0) Xs[buf * (D + 4) + D] = hb;
      more = next();
      if (more) {  // K of the next item, once the value rows of the one before this have been read
        if (c >= 1) mbar_wait_idle(&v_free[buf ^ 1], ((c - 1) >> 1) & 1, status);
        if (lane == 0) load_pair(buf ^ 1, &tmK, &k_full[buf ^ 1], unit, j0);
      }
      mbar_wait_idle(&k_done[buf], (c >> 1) & 1, status);  // every product of this item has read its K tiles
      __syncwarp();
      if (lane == 0) load_pair(buf, &tmV, &v_full[buf], u, first);  // (its arrival publishes X as well)
    }
  } else if (warp == 18) {
    // =============================== copies of Q and the statistics (one lane) ===============================
    if (ptx::elect_one()) {
      int qb = 0;
      while (next()) {
        const float* rstat = last_only ? sc.sstat + (size_t)unit * kTile : sc.stats + (size_t)unit * sc.Mpad;
        for (int rb = 0; rb < nblocks; ++rb, ++qb) {
          const int st = qb % kQStages, ss = qb % kSStages;
          if (qb >= kQStages) mbar_wait_idle(&q_done[st], ((qb / kQStages) - 1) & 1, status);  // the products that read the stage are done
          char* qd = Qst + st * kTB;
          mbar_expect_tx(&q_full[st], kTB);
#pragma unroll
          for (int x = 0; x < kBoxes; ++x) tma_load_2d(qd + x * kHalfBytes, &tmQ, 64 * x, unit * M + rb * kTile, &q_full[st]);
          if (qb >= kSStages) mbar_wait_idle(&st_free[ss], ((qb / kSStages) - 1) & 1, status);  // the stage's last block is summed
          mbar_expect_tx(&st_full[ss], kSF * 4);
          bulk_load(Sst + ss * kSF, rstat + (size_t)rb * kTile, kTile * 4, &st_full[ss]);
          if (kFew) bulk_load(Sst + ss * kSF + kTile, sc.crest + (size_t)unit * kTile, kTile * 4, &st_full[ss]);
        }
      }
    }
  } else if (warp == 16) {
    // =============================== products (one lane) ===============================
    if (ptx::elect_one()) {
      constexpr uint32_t kIdesc = instr_desc(false);
      int qb = 0;
      for (int c = 0; next(); ++c) {
        const int kb = c & 1;
        const uint64_t kd0 = smem_desc(smem_u32(KVs + 2 * kb * kTB), 16, 1024);
        mbar_wait_idle(&k_full[kb], (c >> 1) & 1, status);
        for (int rb = 0; rb < nblocks; ++rb, ++qb) {
          const int buf = qb & 1, st = qb % kQStages;
          mbar_wait_idle(&q_full[st], (qb / kQStages) & 1, status);
          if (qb >= 2) mbar_wait_idle(&c_bar[buf], ((qb - 2) >> 1) & 1, status);  // its S buffers have been read
          tc_fence_after();
          const uint64_t qd0 = smem_desc(smem_u32(Qst + st * kTB), 16, 1024);
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
            for (int ks = 0; ks < kSteps; ++ks)
              umma(tmem + kk * 256 + buf * 128, kd0 + (uint64_t)((kk * kTB) >> 4) + k_major_step(ks), qd0 + k_major_step(ks), kIdesc, ks > 0);
          }
          umma_commit(&s_bar[buf]);
          umma_commit(&q_done[st]);
        }
        umma_commit(&k_done[kb]);
      }
      // (no arrival may still be on its way to this CTA's barriers when the CTA ends)
      if (qb > 0) mbar_wait_idle(&q_done[(qb - 1) % kQStages], ((qb - 1) / kQStages) & 1, status);
    }
  } else {
    // =============================== one key per thread ===============================
    // A thread's 64 rows of a Q block go through registers in four pieces of 16. Two register sets take turns: while
    // one piece is summed, the next piece's logits (TMEM) and statistics (shared memory) are already on their way, so
    // neither latency is waited for. The S buffer is handed back to the products as soon as its last piece is in
    // registers, not when it has been summed.
    const float scale2 = dm.scale * 1.4426950408889634f;
    const int kk = (warp >> 2) & 1, rhalf = tid >> 8, lane = tid & 31, key = tid & (kScoreKeys - 1);
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kk * 256 + rhalf * 64;
    uint32_t va[16], vb[16];
    float4 sa[4], sb[4];
    int qb = 0;
    for (int c = 0; next(); ++c) {
      const int j = j0 + key, need = j - (n - m);  // row R sees key j iff (R % m) >= need
      float h = 0.f, rest_few = 0.f;
      float2 hacc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      auto piece = [&](const uint32_t (&v)[16], const float4 (&st)[4], const float* crest, bool plain, int R0) {
        if constexpr (kFew) score_piece16_few(v, st, crest, scale2, R0, M, m, need, h, rest_few);
        else score_piece16(v, st, scale2, plain, R0, M, m, need, hacc, h);
      };
      mbar_wait(&s_bar[qb & 1], (qb >> 1) & 1, status);
      mbar_wait(&st_full[qb % kSStages], (qb / kSStages) & 1, status);
      tc_fence_after();
      tmem_ld16_issue(t_lane + (qb & 1) * 128, va);
      lds16_issue(Sst + (qb % kSStages) * kSF + rhalf * 64, sa);
      for (int rb = 0; rb < nblocks; ++rb, ++qb) {
        const int buf = qb & 1, ss = qb % kSStages;
        // only the keys of the new block itself are masked (causal inside the block), and only the last
        // row block can have columns beyond M
        const bool plain = (j0 + kScoreKeys - 1 < n - m + 1) && (rb * kTile + kTile <= M);
        const int R0 = rb * kTile + rhalf * 64;
        const uint32_t t_s = t_lane + buf * 128;
        const float* stc = Sst + ss * kSF + rhalf * 64;
        const float* crs = stc + kTile;  // (few only)
        // piece 0 (in va / sa); piece 1 on its way
        tmem_ld16_wait(va);
        tmem_ld16_issue(t_s + 16, vb);
        lds16_issue(stc + 16, sb);
        piece(va, sa, crs, plain, R0);
        // piece 1; piece 2 on its way
        tmem_ld16_wait(vb);
        tmem_ld16_issue(t_s + 32, va);
        lds16_issue(stc + 32, sa);
        piece(vb, sb, crs + 16, plain, R0 + 16);
        // piece 2; piece 3 on its way
        tmem_ld16_wait(va);
        tmem_ld16_issue(t_s + 48, vb);
        lds16_issue(stc + 48, sb);
        piece(va, sa, crs + 32, plain, R0 + 32);
        // piece 3; the S buffer is free, the next block's piece 0 on its way
        tmem_ld16_wait(vb);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&c_bar[buf]);  // this warp holds its part of the S buffer in registers
        if (rb + 1 < nblocks) {
          const int ss1 = (qb + 1) % kSStages;
          mbar_wait(&s_bar[buf ^ 1], ((qb + 1) >> 1) & 1, status);
          mbar_wait(&st_full[ss1], ((qb + 1) / kSStages) & 1, status);  // the next block's row statistics have landed
          tc_fence_after();
          tmem_ld16_issue(t_lane + (buf ^ 1) * 128, va);
          lds16_issue(Sst + ss1 * kSF + rhalf * 64, sa);
        }
        piece(vb, sb, crs + 48, plain, R0 + 48);
        __syncwarp();
        // ... and is done with the block's statistics (no fence: their place is filled again eight blocks later, by a copy that waits
        // for products which wait for all warps to be four blocks further on)
        if (lane == 0) mbar_arrive(&st_free[ss]);
      }
      h += (hacc[0].x + hacc[0].y) + (hacc[1].x + hacc[1].y);

      // ---- c_j = w_j / (1 - w_j) * ||X - v_j||, w_j = h_j / H: the two halves of a key add up ----
      const int kb = c & 1;
      mbar_wait(&v_full[kb], (c >> 1) & 1, status);
      float acc = 0.f;
      {
        // this half's channels of the key's value row: chunks of 8 in the staged tile (boxes of 64 channels, 128-byte swizzle)
        const char* vt = KVs + (2 * kb + (key >> 7)) * kTB;
        const float* x = Xs + kb * (D + 4) + rhalf * (D / 2);
#pragma unroll
        for (int i = 0; i < D / 16; ++i) {
          const uint4 raw = *reinterpret_cast<const uint4*>(vt + tile_off(key & (kTile - 1), rhalf * (D / 16) + i));
          const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float d0 = x[8 * i + 2 * e] - __uint_as_float(w4[e] << 16);
            const float d1 = x[8 * i + 2 * e + 1] - __uint_as_float(w4[e] & 0xffff0000u);
            acc = fmaf(d0, d0, acc);
            acc = fmaf(d1, d1, acc);
          }
        }
      }
      const float hb = kAccum ? Xs[kb * (D + 4) + D] : 0.f;
      fence_async_smem();  // (the rows have been read before the copy that follows the arrival writes there)
      __syncwarp();
      if (lane == 0) mbar_arrive(&v_free[kb]);  // (and with X)
      if (rhalf) {
        hx[kb * kScoreKeys + key] = h;
        ax[kb * kScoreKeys + key] = acc;
        if (kFew) rx[kb * kScoreKeys + key] = rest_few;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kKeyThreads) : "memory");
      if (!rhalf && j < n) {
        h += hx[kb * kScoreKeys + key];
        acc += ax[kb * kScoreKeys + key];
        float rest = kFew ? rest_few + rx[kb * kScoreKeys + key] : (float)M - h;  // (1 - w_j) H
        const size_t slot = (size_t)unit * dm.cap + j;
        if (kAccum) {
          const float bj = base[slot];
          rest += hb - bj;
          h += bj;
          base[slot] = h;
        }
        float ratio = 0.f;
        if (h > 0.f) ratio = (rest > 0.f) ? h / rest : INFINITY;
        scores[slot] = (ratio == 0.f) ? 0.f : ((ratio == INFINITY) ? INFINITY : ratio * sqrtf(acc));
        if (h > kDominant * ((float)M + hb)) {
          sc.dom[2 * unit] = j;
          sc.dom[2 * unit + 1] = __float_as_int(h);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// The score of the token that holds more than kDominant of its unit's weight H (see the file comment), from the others' scores,
// c_i = h_i / (H - h_i) d_i with d_i = || X - v_i ||, so h_i = H c_i / (d_i + c_i). A cluster of kDomCtas CTAs per unit, 512
// threads, a thread one 16-byte piece of every (512 / pieces)-th row of its CTA's share; the shares meet in rank 0 in a fixed
// order. Units without such a token leave at once: what the kernel costs then is its launch, about a microsecond of a step of
// 50 - 60. With one, it is the latency of a few round trips: up to eight rows a thread are fetched before the first is used,
// and before X is known. Block steps without and with one in every unit: 8 units of 4 224 tokens 58.5, 70.4 us (86 with two rows
// in flight and 256 threads); 64 units of 8 320 tokens 640, 750. (As a part of the selection, one CTA per unit and a launch
// less: 58.0 and 95.7, and single-query steps 0.8 % slower for the selection's larger kernel.)
constexpr int kDomCtas = 8, kDomThreads = 512;
template <int D>
__global__ void __launch_bounds__(kDomThreads)
dominant_kernel(Dims dm, const __nv_bfloat16* __restrict__ V, const int* __restrict__ len, Scratch sc, float* scores,
                const float* __restrict__ vsum) {
  constexpr int P = D / 8, kRowsPass = kDomThreads / P, kFly = 8;
  __shared__ __align__(16) float Xs[D + 4], part[kRowsPass][D + 4], mine[D + 4];
  ptx::pdl_wait();
  ptx::pdl_trigger();
  const int unit = blockIdx.x / kDomCtas, rank = (int)ptx::cluster_ctarank(), n = len[unit / dm.Hkv];
  const int slot = sc.dom[2 * unit];
  if (n < dm.m || n > dm.cap || n == 0 || slot < 0) return;  // (the whole cluster)
  const int tid = threadIdx.x, piece = tid % P, g = tid / P;
  const uint4* src = reinterpret_cast<const uint4*>(V + (size_t)unit * dm.cap * D) + piece;
  const float* cu = scores + (size_t)unit * dm.cap;
  const int share = (n + kDomCtas - 1) / kDomCtas, r0 = rank * share, r1 = min(n, r0 + share);
  uint4 raw[kFly];
  float c[kFly];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int j = j0 + u * kRowsPass;
      raw[u] = j < r1 ? src[(size_t)j * P] : make_uint4(0u, 0u, 0u, 0u);
      c[u] = j < r1 && j != slot ? cu[j] : 0.f;
    }
  };
  auto unpack = [](uint4 r, float (&v)[8]) {
    const uint32_t x[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      v[2 * e] = __uint_as_float(x[e] << 16);
      v[2 * e + 1] = __uint_as_float(x[e] & 0xffff0000u);
    }
  };
  int at = r0 + g;
  fetch(at);
  const uint4 top = src[(size_t)slot * P];
  if (tid < 32) {
    float x[D / 32];
    const float hb = x_from_parts<D>(dm, sc, unit, n, vsum, tid, x);
#pragma unroll
    for (int i = 0; i < D / 32; ++i) Xs[tid * (D / 32) + i] = x[i];
    if (tid == 0) Xs[D] = hb;
  }
  __syncthreads();
  const float H = (float)sc.Ms + Xs[D];
  float vt[8], w[8], xp[8], S = 0.f;
  unpack(top, vt);
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    w[e] = 0.f;
    xp[e] = Xs[8 * piece + e];
  }
  for (int j0 = r0; j0 < r1; j0 += kFly * kRowsPass) {  // (the same rounds for every thread: its shuffles are the warp's)
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      float v[8], d2 = 0.f;
      unpack(raw[u], v);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float d = xp[e] - v[e];
        d2 = fmaf(d, d, d2);
      }
#pragma unroll
      for (int o = 1; o < P; o <<= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      const float h = c[u] > 0.f ? H * (c[u] / (sqrtf(d2) + c[u])) : 0.f;
      S += h;
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = fmaf(h, v[e] - vt[e], w[e]);
    }
    at += kFly * kRowsPass;
    fetch(at);
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) part[g][8 * piece + e] = w[e];
  if (piece == 0) part[g][D] = S;
  __syncthreads();
  if (tid <= D) {
    float t = 0.f;
#pragma unroll 8
    for (int i = 0; i < kRowsPass; ++i) t += part[i][tid];
    mine[tid] = t;
  }
  ptx::cluster_sync_all();
  if (rank == 0 && tid <= D) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < kDomCtas; ++i) t += ptx::ld_dsmem_f32(ptx::map_to_rank(ptx::smem_u32(mine + tid), i));
    part[0][tid] = t;
  }
  ptx::cluster_sync_all();  // (nobody leaves while its share is read)
  if (rank == 0 && tid < 32) {
    float d2 = 0.f;
#pragma unroll
    for (int ch = tid; ch < D; ch += 32) {
      const float d = vsum ? Xs[ch] - __bfloat162float(V[((size_t)unit * dm.cap + slot) * D + ch]) : part[0][ch] / H;
      d2 = fmaf(d, d, d2);
    }
    d2 = warp_sum(d2);
    if (tid == 0) {
      const float rest = part[0][D];
      scores[(size_t)unit * dm.cap + slot] = rest > 0.f ? __int_as_float(sc.dom[2 * unit + 1]) / rest * sqrtf(d2) : INFINITY;
    }
  }
}

// The scores when the caller supplies the weights (EXTERNAL): h_j = base_j, one pass over V. grid = (ceil(cap / kExtKeys),
// units): four threads per token, D / 4 channels each.
constexpr int kExtKeys = 128;
template <int D>
__global__ void __launch_bounds__(4 * kExtKeys)
score_external_kernel(Dims dm, const __nv_bfloat16* __restrict__ V, const int* __restrict__ len, Scratch sc,
                      const float* __restrict__ base, float* __restrict__ scores, const float* __restrict__ vsum) {
  __shared__ __align__(16) float Xs[D + 4];
  ptx::pdl_wait();
  ptx::pdl_trigger();
  const int unit = blockIdx.y, n = len[unit / dm.Hkv], j = blockIdx.x * kExtKeys + (threadIdx.x >> 2), part = threadIdx.x & 3;
  if (n < dm.m || n > dm.cap || blockIdx.x * kExtKeys >= n) return;
  if (threadIdx.x < 32) {
    float xr[D / 32];
    const float hb = x_from_parts<D>(dm, sc, unit, n, vsum, threadIdx.x, xr);
#pragma unroll
    for (int i = 0; i < D / 32; ++i) Xs[threadIdx.x * (D / 32) + i] = xr[i];
    if (threadIdx.x == 0) Xs[D] = hb;
  }
  __syncthreads();
  float acc = 0.f;
  if (j < n) {
    const uint4* row = reinterpret_cast<const uint4*>(V + ((size_t)unit * dm.cap + j) * D);
    const float4* x = reinterpret_cast<const float4*>(Xs);
#pragma unroll
    for (int i = 0; i < D / 32; ++i) {  // the four threads' chunks of 8 channels side by side
      const int c = 4 * i + part;
      const uint4 raw = row[c];
      const float4 a = x[2 * c], b = x[2 * c + 1];
      const float d0 = a.x - __uint_as_float(raw.x << 16), d1 = a.y - __uint_as_float(raw.x & 0xffff0000u);
      const float d2 = a.z - __uint_as_float(raw.y << 16), d3 = a.w - __uint_as_float(raw.y & 0xffff0000u);
      const float d4 = b.x - __uint_as_float(raw.z << 16), d5 = b.y - __uint_as_float(raw.z & 0xffff0000u);
      const float d6 = b.z - __uint_as_float(raw.w << 16), d7 = b.w - __uint_as_float(raw.w & 0xffff0000u);
      acc = fmaf(d0, d0, fmaf(d1, d1, fmaf(d2, d2, fmaf(d3, d3, acc))));
      acc = fmaf(d4, d4, fmaf(d5, d5, fmaf(d6, d6, fmaf(d7, d7, acc))));
    }
  }
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  if (part == 0 && j < n) {
    const size_t slot = (size_t)unit * dm.cap + j;
    const float h = base[slot], rest = Xs[D] - h;
    const float ratio = h > 0.f ? (rest > 0.f ? h / rest : INFINITY) : 0.f;
    scores[slot] = (ratio == 0.f) ? 0.f : ((ratio == INFINITY) ? INFINITY : ratio * sqrtf(acc));
  }
}

}  // namespace prefill
}  // namespace caote
