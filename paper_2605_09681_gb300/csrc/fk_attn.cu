// Chunk attention over the per-head packed views (Sec. 4.2 Eq. 2, Sec. 4.3 Eq. 4):
// O = softmax(Q K^T / sqrt(D)) V per head, with a different key count per head.
//
// One CTA computes two 128-row query tiles of one head (small grids: one, over two sets of keys, see
// kOne) against all of the head's keys, in tiles of 128 keys, on the 5th-generation tensor cores:
//   warp 8 (one lane)  TMA: both Q tiles once (3D map over [Nq][H][D]), K and V tiles (2D
//                      maps over the view arenas) into two-stage rings, 128-byte swizzle;
//                      key tile 0 on its own barrier, then V_j together with K_{j+1} on one
//                      barrier per stage pair (one wait and one release per key tile);
//   warp 9             tcgen05.mma, per key tile j and query tile t: P_t V_j of keys 0-95, of
//                      keys 96-127 (each once its P is in TMEM), then S_t(j+1)
//                      (S_t = Q_t K^T into TMEM, O_t += P_t V with P_t read from TMEM);
//                      completion via tcgen05.commit; the warp stays converged and an elected
//                      lane issues (see elect_one);
//   warps 0-3 / 4-7    softmax of query tile 0 / 1 (ping-pong: one warpgroup's softmax
//                      overlaps the other tile's MMAs): thread r owns row r = TMEM lane r,
//                      reads S with tcgen05.ld, online softmax in the log2 domain with a
//                      lazily raised running max, writes P as bf16 pairs over S columns already
//                      read with tcgen05.st, and finally normalises O and stores it.  A key tile
//                      goes to the MMA warp in two parts, keys 0-95 and 96-127, so that P V of the
//                      first runs while the second is computed.  After the first key tile a part's
//                      P is computed with the running max at once; its sum (at most 2^8) shows
//                      that no numerator exceeds that bound, else the part is done again with
//                      a max pass that raises the running max and rescales O and the row sum.
//                      What bounds it (clock64 timeline of one CTA, 12 heads x 25480 keys, D =
//                      128): one key tile takes ~2450 cycles for 2048 cycles of MMA; a tile's
//                      softmax takes ~1090 of them and its P waits ~500 for the tensor pipe.  One
//                      hand-over per tile, a vote and a store wait per 64 columns and S kept for
//                      both took 1230; a denoising step at 480P then ran 321 us (303 in two parts,
//                      298 with the shorter waits since), a step under FP8 Q K^T 326 us (289; 276), a
//                      1080P step 6.22 ms (5.57; 5.51).  96 + 32: P V of the first part (384 cycles)
//                      covers the second's arithmetic (~190).
// TMEM columns: S0 0-127, S1 128-255, O0 256.., O1 256+D.. (512 allocated).
// FP8_QK variant (D = 128): the K tiles hold E4M3 codes (one 128-byte swizzle atom per row,
// from the view arena's E4M3 copy); the bf16 Q tiles are loaded as usual and each softmax
// thread quantizes its own row into an E4M3 tile (row exponent e_row, codes of the row times
// 2^-e_row, written in the 128-byte swizzle pattern) before the first MMA; S = Q K^T runs as
// tcgen05.mma kind::f8f6f4 (K = 32 per instruction) and the thread scales its row's logits by
// 2^e_row along with 1/sqrt(D); P V is unchanged (bf16).
// FP8 variant (P V too): the V tiles hold E4M3 codes of the V arena's E4M3 copy, P is stored
// as E4M3 codes of 2^6 exp2(S c - m) (four per TMEM column) with m an integer running
// reference, and P V runs as kind::f8f6f4; O and the row sum are rescaled by exact powers of
// two when the reference moves.
// Every mbarrier wait is bounded (%globaltimer); on expiry the CTA records
// FK_ERR_TIMEOUT in the status word, drains its own TMA loads and MMAs and frees TMEM.
// The kernel is launched with programmatic dependent launch: its setup (barriers, TMEM) may
// overlap the tail of the kernel before it in the stream (the compaction or current-chunk
// kernel, which write the K/V views, or whatever kernel produced Q), and the TMA thread waits
// for that kernel (griddepcontrol.wait) before its first load; every global write of this
// kernel follows MMAs that consume those loads.  It never triggers its own dependents early.
#include "fk_internal.h"

namespace fk {
namespace {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s per wait
constexpr float kRescaleThreshold = 1.0f;          // log2 units: a part that exceeds the bound raises m
// FP8 P V: P is stored as e4m3 of 2^6 exp2(s c - m), m an integer running reference (the running
// max rounded up) that lags the row max by less than log2(432) - 6 = 2.76, so that a stored code is at
// most 416 (with a bound of 2^8 m was raised, and O rescaled, so much more often that a 480P launch
// took 261 us and not 241); reference changes rescale O and l by exact powers of two
constexpr float kRescaleThresholdFp8 = 2.0f;
constexpr float kPShiftFp8 = 6.0f;
// Running maximum (log2 domain) before any key.  Finite: keys whose logits are all -inf (products
// below the float range) then give numerators exp2(-inf) = 0 and not exp2(-inf + inf) = NaN, also where
// they fill all that one key split or key set begins with; the first finite logit raises it, with alpha = 0.
constexpr float kNoMax = -3.402823466e38f;

constexpr int kWarpTma = 8;                        // warps 0-3 / 4-7: softmax of query tile 0 / 1
constexpr int kWarpMma = 9;
constexpr int kAttnThreads = 320;

struct AttnBarriers {
  uint64_t q_full;
  uint64_t k_full[2], k_empty[2];   // profiling: the key ring
  uint64_t k0_full, k0_empty;       // attention: key tile 0 (stage 0)
  uint64_t vk_full[2], vk_empty[2]; // attention, b = j mod 2: V_j (V stage b) with K_{j+1} (K stage 1-b)
  uint64_t s_full[2], p_full[2];
  uint64_t pa_full[2], pva_done[2];  // attention: P of a tile's first 96 keys written / multiplied
  uint64_t o_done, fin;
  uint64_t q8_ready;            // FP8_QK: the 256 softmax threads have written the E4M3 Q rows
  uint32_t tmem_base;
  volatile int abort;
};

template <int D, bool kFp8 = false, bool kFp8PV = false>
struct Layout {
  static constexpr int kQ = kAttnBM * D * (kFp8 ? 1 : 2);   // one 128-row query tile (MMA operand)
  static constexpr int kK = kAttnBN * D * (kFp8 ? 1 : 2);   // one 128-key K tile
  static constexpr int kKV = kAttnBN * D * (kFp8PV ? 1 : 2);  // one 128-key V tile
  static constexpr int kQ16 = kFp8 ? kAttnBM * D * 2 : 0;   // FP8: one bf16 query tile as loaded
  static constexpr int kOffQ = 0;                 // two query tiles
  static constexpr int kOffK = kOffQ + 2 * kQ;    // two K stages
  static constexpr int kOffV = kOffK + 2 * kK;    // two V stages
  static constexpr int kOffQ16 = kOffV + 2 * kKV; // FP8: two bf16 query tiles
  static constexpr int kOffBar = kOffQ16 + 2 * kQ16;
  static constexpr int kUsed = kOffBar + 256;
  // the merge's rows of O (256, or 128 and the exchange of as many bytes), their (m, l) and, with one query
  // tile per CTA, the two key sets' own
  static_assert(2 * kAttnBM * D * 4 + 3 * kAttnBM * 8 <= kOffBar, "the merge leaves the barriers alone");
  // at least ~116 KB so that one CTA occupies an SM (its 512 TMEM columns are then free)
  static constexpr int kSmem = (kUsed + 1024) > 118 * 1024 ? (kUsed + 1024) : 118 * 1024;
};

__device__ __forceinline__ uint32_t su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(su32(b)),
               "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(su32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"

      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait for the phase of parity `parity`.  Returns false when the CTA is
// aborting or the limit expired (which starts the abort).  Inlined: a call would save and
// restore the caller's live registers on every wait, even when the phase is complete.
__device__ __forceinline__ bool wait_phase(uint64_t* b, uint32_t parity, AttnBarriers* bar,
                                           int* status, bool honour_abort = true) {
  if (mbar_test(b, parity)) return true;
  const uint64_t t0 = now_ns();
  while (true) {
    if (mbar_test(b, parity)) return true;
    if (honour_abort && bar->abort) return false;
    if (now_ns() - t0 > kWaitLimitNs) {
      bar->abort = 1;
      atomicOr(status, kStatusTimeout);
      return false;
    }
  }
}

// Warp-uniform bounded wait: every lane polls and every poll is a decision of the warp, with the
// abort flag and the clock looked at on each 16th (a wait per lane and one vote at the end cost 2-3%
// of an attention launch; polls that do not suspend, test_wait, 8%).
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, AttnBarriers* bar,
                                          int* status) {
  if (__all_sync(0xffffffffu, mbar_test(b, parity))) return true;
  const uint64_t t0 = now_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 16; ++i)
      if (__all_sync(0xffffffffu, mbar_test(b, parity))) return true;
    bool stop = bar->abort;
    if (now_ns() - t0 > kWaitLimitNs) {
      bar->abort = 1;
      atomicOr(status, kStatusTimeout);
      stop = true;
    }
    if (__any_sync(0xffffffffu, stop)) return false;
  }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* b,
                                            int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];"
      :: "r"(su32(dst)), "l"(map), "r"(su32(b)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* b,
                                            int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      :: "r"(su32(dst)), "l"(map), "r"(su32(b)), "r"(x), "r"(y), "r"(z) : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor (tcgen05): start, leading/stride byte offsets (16-byte
// units), descriptor version 1, 128-byte swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}

// Instruction descriptor, kind::f16: f32 accumulate, bf16 A and B, A K-major,
// B K-major (b_mn = 0) or MN-major (b_mn = 1), N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// Instruction descriptor, kind::f8f6f4: f32 accumulate, A and B E4M3 (type code 0 at bits
// 7 and 10), A K-major, B K-major (b_mn = 0) or MN-major (b_mn = 1).
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N, int b_mn = 0) {
  return (1u << 4) | ((uint32_t)b_mn << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One lane of the (converged) warp, the same one each time.  tcgen05.mma and commit behind this
// predicate take their operands from uniform registers; behind `lane == 0` the compiler does not
// know that one lane is left, and an MMA cost 80-100 cycles of issue whatever its size.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e != 0;
}

__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                     uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]: A (M x 16, bf16 pairs packed along 8 columns) in tensor memory
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      :: "r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T on E4M3 operands (both K-major, K = 32 per instruction)
__device__ __forceinline__ void umma_f8(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n"
      :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem] on E4M3 operands: A (M x 32, four codes per 32-bit column) in
// tensor memory, B from a shared-memory descriptor
__device__ __forceinline__ void umma_ts_f8(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}\n"
      :: "r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* b) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
      :: "r"(su32(b)) : "memory");
}

#define FK_TMEM_LD32(taddr, v)                                                              \
  asm volatile(                                                                             \
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"  \
      "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];" \
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),  \
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),           \
        "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),        \
        "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),        \
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),        \
        "=r"(v[31])                                                                         \
      : "r"(taddr))

#define FK_TMEM_ST32(taddr, v)                                                              \
  asm volatile(                                                                             \
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"   \
      "%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" \
      :: "r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),      \
        "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]),      \
        "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]),  \
        "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),  \
        "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory")

#define FK_TMEM_ST8(taddr, v)                                                               \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"     \
               :: "r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]),        \
               "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory")

#define FK_TMEM_ST16(taddr, v)                                                              \
  asm volatile(                                                                             \
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"   \
      "%12,%13,%14,%15,%16};"                                                               \
      :: "r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),      \
        "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]),      \
        "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory")

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// barrier over every thread of the cluster (release / acquire)
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
// shared-memory address of CTA `rank` of the cluster, and loads from such an address
__device__ __forceinline__ uint32_t map_peer(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_peer4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_peer2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

// packed fp32 pair arithmetic (sm_100+): two lanes of work per instruction
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " mov.b64 rc, {%6, %7};\n fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " add.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// four non-negative floats -> four E4M3 codes (lowest key in the low byte)
__device__ __forceinline__ uint32_t e4m3x4(float2 a, float2 b) {
  uint32_t w;
  asm("{\n .reg .b16 lo, hi;\n cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n"
      " cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n mov.b32 %0, {lo, hi};\n}"
      : "=r"(w) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return w;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// tcgen05.wait::ld that also names the registers of the loads it completes, so that no use of
// them can be scheduled before it
#define FK_TMEM_WAIT_LD32(v)                                                                \
  asm volatile("tcgen05.wait::ld.sync.aligned;"                                             \
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),    \
                 "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),  \
                 "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]),           \
                 "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]),           \
                 "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]),           \
                 "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])            \
               :: "memory")

// 32-column chunks `first` .. `first` + `count` - 1 of a key tile
template <int kFirst, int kCount>
struct Chunks {
  static constexpr int first = kFirst, count = kCount;
};

// 32 logits -> numerators exp2(s * sc + nm): their sums in four chains, and P words (bf16 pairs, or
// four E4M3 codes; `ov` then collects the bits of the overflow test).  The sums and roundings of a
// pair come kSkew pairs after its exponentials, so that they do not wait for them.
constexpr int kSkew = 4;
template <bool kE4m3>
__device__ __forceinline__ void exp_chunk(const uint32_t* s, float2 sc2, float2 nm2, float2* ah,
                                          uint32_t* pk, uint32_t& ov) {
  float2 e[16];
#pragma unroll
  for (int q = 0; q < 16 + kSkew; ++q) {
    if (q < 16) {
      const float2 x = ffma2(make_float2(__uint_as_float(s[2 * q]), __uint_as_float(s[2 * q + 1])), sc2, nm2);
      e[q] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
    }
    if (q >= kSkew) {
      const int p = q - kSkew;
      ah[p & 3] = fadd2(ah[p & 3], e[p]);
      if constexpr (kE4m3) {
        if (p & 1) {
          pk[p >> 1] = e4m3x4(e[p - 1], e[p]);
          ov |= pk[p >> 1] + 0x02020202u;
        }
      } else {
        pk[p] = pack_bf16(e[p].x, e[p].y);
      }
    }
  }
}

// 32 logits -> the sums of exp2(s * sc + nm) in four chains
__device__ __forceinline__ void exp_sum(const uint32_t* s, float2 sc2, float2 nm2, float2* ah) {
  float2 e[16];
#pragma unroll
  for (int q = 0; q < 16 + kSkew; ++q) {
    if (q < 16) {
      const float2 x = ffma2(make_float2(__uint_as_float(s[2 * q]), __uint_as_float(s[2 * q + 1])), sc2, nm2);
      e[q] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
    }
    if (q >= kSkew) ah[q & 3] = fadd2(ah[q & 3], e[q - kSkew]);
  }
}

// Whether a numerator of these columns may exceed the bound in any lane (warp-uniform).  bf16, 2^8: no more
// than their sum does.  E4M3 (the bound is then 432, the values that round above 416 or saturate):
// exactly when a code is 0x7E; codes are non-negative and at most 0x7E, so adding 2 to each byte sets
// its top bit then, without carries between bytes.
template <bool kE4m3>
__device__ __forceinline__ bool exceeds(const float2* ah, uint32_t ov) {
  if constexpr (kE4m3) return __any_sync(0xffffffffu, (ov & 0x80808080u) != 0);
  const float2 hs2 = fadd2(fadd2(ah[0], ah[1]), fadd2(ah[2], ah[3]));
  return __any_sync(0xffffffffu, hs2.x + hs2.y > 256.0f);
}

// Rows [g0, g0 + rows) of the key splits' merge by one of 8 warps: with M = max_s m_s (log2 domain),
// O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s as bf16, `stride` elements from row to row.  D / 4
// lanes read a row, 16 bytes each; lane k first forms the S <= kS weights of the warp's k-th row.  A
// load from a peer takes 600-900 cycles, so every split's (and kRows row groups') are in flight; more of
// them cost more in instruction fetch than they hide (the code runs once per CTA).
template <int D, int kS, int kRows>
__device__ __forceinline__ void merge_rows(uint32_t part, uint32_t ml, int S, int g0, int rows, bf16* O, int stride,
                                           int warp, int lane) {
  constexpr int kLanes = D / 4, kSub = 32 / kLanes;
  const int sub = lane / kLanes, li = lane % kLanes;
  float4 x[kRows][kS];
  auto load = [&](int i0) {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = ((i0 + i) * 8 + warp) * kSub + sub;
      const uint32_t addr = part + (uint32_t)((g0 + r) * (D * 4) + li * 16);
#pragma unroll
      for (int sp = 0; sp < kS; ++sp)
        x[i][sp] = r < rows && sp < S ? ld_peer4(map_peer(addr, sp)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
  };
  load(0);
  float w[kS];
  {
    const int r = ((lane / kSub) * 8 + warp) * kSub + lane % kSub;
    float2 e[kS];
    float M = -INFINITY, L = 0.0f;
#pragma unroll
    for (int sp = 0; sp < kS; ++sp)
      e[sp] = r < rows && sp < S ? ld_peer2(map_peer(ml + (uint32_t)((g0 + r) * 8), sp)) : make_float2(-INFINITY, 0.0f);
#pragma unroll
    for (int sp = 0; sp < kS; ++sp) M = fmaxf(M, e[sp].x);
#pragma unroll
    for (int sp = 0; sp < kS; ++sp) {
      w[sp] = sp < S ? fast_exp2(e[sp].x - M) : 0.0f;
      L = fmaf(w[sp], e[sp].y, L);
    }
    const float inv = 1.0f / L;
#pragma unroll
    for (int sp = 0; sp < kS; ++sp) w[sp] *= inv;
  }
#pragma unroll 1
  for (int i0 = 0; (i0 * 8 + warp) * kSub < rows; i0 += kRows) {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = ((i0 + i) * 8 + warp) * kSub + sub;
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int sp = 0; sp < kS; ++sp) {
        const float ws = __shfl_sync(0xffffffffu, w[sp], ((i0 + i) * kSub + sub) & 31);
        acc.x = fmaf(ws, x[i][sp].x, acc.x);
        acc.y = fmaf(ws, x[i][sp].y, acc.y);
        acc.z = fmaf(ws, x[i][sp].z, acc.z);
        acc.w = fmaf(ws, x[i][sp].w, acc.w);
      }
      if (r < rows)
        *reinterpret_cast<uint2*>(O + (int64_t)r * stride + (li ^ ((g0 + r) & (D / 4 - 1))) * 4) =
            make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
    }
    load(i0 + kRows);
  }
}

// kSplit: a launch with key splits (kv_splits > 1): the splits of one pair of query tiles are the
// CTAs of a cluster, merged at the end through distributed shared memory.  kFp8: Q K^T on E4M3
// operands (D = 128).  kFp8PV (with kFp8): P V on E4M3 operands too: V tiles from the E4M3 copy of
// the V view arena (one 128-byte swizzle atom per key row), P written as e4m3 of 2^6 exp2(s c - m),
// four keys per TMEM column.
// kOne: one query tile per CTA, so that a small grid has twice the CTAs and a cluster half the rows to
// merge: both warpgroups own the same rows, warpgroup t over key tiles t, t + 2, .. (the two sets of S,
// P and O in tensor memory are the key sets' instead of the query tiles'), merged at the end like two
// more splits.  Per key tile a CTA takes 0.65 of the time for twice the K and V per query (when it pays:
// choose_attention_plan).  6 heads, 808 queries, 2828 and 2020 keys, D = 128: 16.8 -> 14.3 us a launch.
template <int D, bool kSplit, bool kFp8, bool kFp8PV = false, bool kOne = false>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
            const __grid_constant__ CUtensorMap tmV, const AttnArgs a) {
  static_assert(!kFp8 || D == 128, "FP8_QK: one 128-byte swizzle atom per Q / K row");
  static_assert(!kFp8PV || kFp8, "FP8 P V comes with FP8 Q K^T");
  static_assert(!kOne || kSplit, "the two key sets' merge is the key splits' one");
  using Lay = Layout<D, kFp8, kFp8PV>;
  constexpr float kThr = kFp8PV ? kRescaleThresholdFp8 : kRescaleThreshold;
  constexpr float kPShift = kFp8PV ? kPShiftFp8 : 0.0f;
  constexpr int kHalves = D / 64;                 // 64-column (128-byte) swizzle atoms
  // S_t(j + kAhead) follows P_t V_j; a query tile's (kOne: key set's) first key tile is below kAhead
  constexpr int kAhead = kOne ? 2 : 1;
  constexpr uint32_t kTmemCols = 512;
  constexpr uint32_t kColO = 2 * kAttnBN;         // S0 = cols 0..127, S1 = 128..255, O0, O1 after
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* sQ = smem + Lay::kOffQ;
  uint8_t* sK = smem + Lay::kOffK;
  uint8_t* sV = smem + Lay::kOffV;
  uint8_t* sQ16 = smem + Lay::kOffQ16;            // FP8: bf16 query tiles (TMA destination)
  AttnBarriers* bar = reinterpret_cast<AttnBarriers*>(smem + Lay::kOffBar);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // CTA = (head slot, pair of query tiles, key split).  Split `split` of kv_splits covers key
  // tiles [j0, j1) of the head: the CTA sees it as a head of nk keys starting at row0.
  const int split = kSplit ? blockIdx.x % a.kv_splits : 0;
  const int rest = kSplit ? blockIdx.x / a.kv_splits : blockIdx.x;
  const int hi = rest / a.n_qtiles;
  const int q0 = (rest - hi * a.n_qtiles) * ((kOne ? 1 : 2) * kAttnBM);
  const int head = a.head_of[hi];
  int nk = a.n_keys[head];
  int row0 = a.row_base[head];
  if constexpr (kSplit) {
    const int nt_head = (nk + kAttnBN - 1) / kAttnBN;
    const int j0 = split * nt_head / a.kv_splits, j1 = (split + 1) * nt_head / a.kv_splits;
    nk = min(nk, j1 * kAttnBN) - j0 * kAttnBN;
    row0 += j0 * kAttnBN;
  }
  const int nt = (nk + kAttnBN - 1) / kAttnBN;

  // The TMA warp makes the barriers and starts Q and K tile 0 before the CTA meets (the tensor
  // memory allocation takes ~1000 cycles).
  constexpr int kQBytes = kAttnBM * D * 2;
  auto load_k = [&](int j, uint64_t* b) {             // key tile j into K stage j mod 2
    const int st = j & 1;
    if constexpr (kFp8) {
      tma_load_2d(sK + st * Lay::kK, &tmK, b, 0, row0 + j * kAttnBN);
    } else {
      for (int h = 0; h < kHalves; ++h)
        tma_load_2d(sK + st * Lay::kK + h * 16384, &tmK, b, h * 64, row0 + j * kAttnBN);
    }
  };
  if (warp == kWarpTma && lane == 0) {
    mbar_init(&bar->q_full, 1);
    mbar_init(&bar->k0_full, 1);
    mbar_init(&bar->k0_empty, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar->vk_full[i], 1);
      mbar_init(&bar->vk_empty[i], 1);
      mbar_init(&bar->s_full[i], 1);
      mbar_init(&bar->p_full[i], 4);
      mbar_init(&bar->pa_full[i], 4);
      mbar_init(&bar->pva_done[i], 1);
    }
    mbar_init(&bar->o_done, 1);
    mbar_init(&bar->fin, 1);
    if (kFp8) mbar_init(&bar->q8_ready, (kOne ? 1 : 2) * kAttnBM);
    bar->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // Q, K and V may have been written by the previous kernel of the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // bf16 query tiles: the MMA operand, or (FP8) the softmax threads' quantization input
    uint8_t* q_dst = kFp8 ? sQ16 : sQ;
    mbar_expect_tx(&bar->q_full, (kOne ? 1 : 2) * kQBytes);
    for (int t = 0; t < (kOne ? 1 : 2); ++t)
      for (int h = 0; h < kHalves; ++h)
        tma_load_3d(q_dst + t * kQBytes + h * 16384, &tmQ, &bar->q_full, h * 64, head, q0 + t * kAttnBM);
    const bool k1 = kOne && nt > 1;                 // kOne: key tiles 0 and 1
    mbar_expect_tx(&bar->k0_full, (k1 ? 2 : 1) * Lay::kK);
    load_k(0, &bar->k0_full);
    if (k1) load_k(1, &bar->k0_full);
  }
  __syncwarp();
  if (warp == kWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(su32(&bar->tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;

  if (warp == kWarpTma) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int lastVK[2] = {-1, -1};
      bool ok = true;
      // per key tile j: V_j together with K_{j+1} on one barrier (b = j mod 2).  Their
      // stages were last used by V_{j-2} and K_{j-1}, released together by vk_empty[b] after
      // iteration j-2's MMAs (K_2 reuses K_0's stage: k0_empty).  kOne: V_j with K_{j+2}, whose stage
      // K_j leaves with iteration j-2 (tiles 0 and 1: k0_empty).
      for (int j = 0; j < nt && ok; ++j) {
        const int bb = j & 1, u = j >> 1;
        const bool more = j + kAhead < nt;
        if (j >= 2 && !wait_phase(&bar->vk_empty[bb], (u - 1) & 1, bar, a.status)) { ok = false; break; }
        if (!kOne && j == 1 && more && !wait_phase(&bar->k0_empty, 0, bar, a.status)) { ok = false; break; }
        mbar_expect_tx(&bar->vk_full[bb], Lay::kKV + (more ? Lay::kK : 0));
        if constexpr (kFp8PV) {
          tma_load_2d(sV + bb * Lay::kKV, &tmV, &bar->vk_full[bb], 0, row0 + j * kAttnBN);
        } else {
          for (int h = 0; h < kHalves; ++h)
            tma_load_2d(sV + bb * Lay::kKV + h * 16384, &tmV, &bar->vk_full[bb], h * 64,
                        row0 + j * kAttnBN);
        }
        lastVK[bb] = u;
        if (kOne && j < 2 && more && !wait_phase(&bar->k0_empty, 0, bar, a.status)) { ok = false; break; }
        if (more) load_k(j + kAhead, &bar->vk_full[bb]);
      }
      if (!ok) {   // drain every load this thread issued before the CTA exits
        wait_phase(&bar->q_full, 0, bar, a.status, false);
        wait_phase(&bar->k0_full, 0, bar, a.status, false);
        for (int bb = 0; bb < 2; ++bb)
          if (lastVK[bb] >= 0) wait_phase(&bar->vk_full[bb], lastVK[bb] & 1, bar, a.status, false);
      }
    }
    __syncwarp();
    if constexpr (kSplit) {                        // the merge's two barriers
      cluster_sync();
      cluster_sync();
    }
  } else if (warp == kWarpMma) {
    // ------------------------------------------------------------------ MMA issuer
    // Order per key tile j:  PV0(j), S0(j+1), PV1(j), S1(j+1).  Tensor-core operations of
    // one thread complete in issue order, so when S_t(j+1) is reported complete, PV_t(j)
    // is complete too: the softmax of tile j+1 may rescale O_t without a further wait, and
    // S_t(j+1) overwriting P_t(j) (same columns) happens after PV_t(j) has read it.
    // kOne: PV_t(j), S_t(j+2) with t = j mod 2.
    constexpr uint32_t kIdQK = kFp8 ? idesc_e4m3(kAttnBM, kAttnBN) : idesc_bf16(kAttnBM, kAttnBN, 0);
    constexpr uint32_t kIdPV = kFp8PV ? idesc_e4m3(kAttnBM, D, 1) : idesc_bf16(kAttnBM, D, 1);
    const uint64_t dQ = sdesc(su32(sQ), 16, 1024), dK = sdesc(su32(sK), 16, 1024);
    const uint64_t dV = sdesc(su32(sV), 16384, 1024);
    auto qk = [&](int j, int t) {
      const uint64_t da = dQ + (uint32_t)((kOne ? 0 : t) * (Lay::kQ >> 4)), db = dK + (uint32_t)((j & 1) * (Lay::kK >> 4));
      const uint32_t d = tmem + (uint32_t)(t * kAttnBN);
      if constexpr (kFp8) {
        // 128 codes per row = one swizzle atom: four K = 32 steps of 32 bytes
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) umma_f8(d, da + kk * 2, db + kk * 2, kIdQK, kk > 0 ? 1u : 0u);
      } else {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (uint32_t)((kk >> 2) * 1024 + (kk & 3) * 2);
          umma(d, da + off, db + off, kIdQK, kk > 0 ? 1u : 0u);
        }
      }
      umma_commit(&bar->s_full[t]);
    };
    // PV of a tile's keys 32 c0 .. 32 c1 - 1
    auto pv = [&](int j, int t, int c0, int c1) {
      const uint64_t db = dV + (uint32_t)((j & 1) * (Lay::kKV >> 4));
      const uint32_t d = tmem + kColO + (uint32_t)(t * D), p = tmem + (uint32_t)(t * kAttnBN);
      if constexpr (kFp8PV) {
        // 32 keys per step: P columns 8 kk .. 8 kk + 7 (four codes each); V rows 32 kk .. +31,
        // MN-major (d contiguous, 128 bytes per key row), 8-row groups 1024 bytes apart
#pragma unroll
        for (int kk = c0; kk < c1; ++kk)
          umma_ts_f8(d, p + kk * 8, db + kk * 256, kIdPV, (j >= kAhead || kk > 0) ? 1u : 0u);
      } else {
#pragma unroll
        for (int kk = 2 * c0; kk < 2 * c1; ++kk)
          umma_ts(d, p + kk * 8, db + kk * 128, kIdPV, (j >= kAhead || kk > 0) ? 1u : 0u);
      }
    };
    // every lane waits, one issues: the warp stays converged
    auto wait = [&](uint64_t* b, uint32_t parity) { return warp_wait(b, parity, bar, a.status); };
    bool ok = wait(kFp8 ? &bar->q8_ready : &bar->q_full, 0) && wait(&bar->k0_full, 0);
    if (ok) {
      tc_fence_after();
      if (elect_one()) {
        qk(0, 0);
        if (!kOne) qk(0, 1);
        else if (nt > 1) qk(1, 1);
        umma_commit(&bar->k0_empty);
      }
    }
    for (int j = 0; j < nt && ok; ++j) {
      const int bb = j & 1;
      const bool more = j + kAhead < nt;
      const uint32_t ph = kOne ? (j >> 1) & 1 : j & 1;   // of a query tile's (kOne: key set's) barriers
      // V_j and K_{j+1} (one barrier) before P_0(j): neither depends on the softmax, and
      // PV0(j), S0(j+1) then go to the tensor pipe back to back once P_0(j) is in TMEM
      if (!wait(&bar->vk_full[bb], (j >> 1) & 1)) { ok = false; break; }
#pragma unroll
      for (int i = 0; i < (kOne ? 1 : 2); ++i) {
        const int t = kOne ? bb : i;
        if (!wait(&bar->pa_full[t], ph)) { ok = false; break; }
        tc_fence_after();
        if (elect_one()) {
          pv(j, t, 0, 3);
          umma_commit(&bar->pva_done[t]);
        }
        if (!wait(&bar->p_full[t], ph)) { ok = false; break; }
        tc_fence_after();
        if (elect_one()) {
          pv(j, t, 3, 4);
          if (more) qk(j + kAhead, t);
          if (kOne || t == 1) umma_commit(&bar->vk_empty[bb]);   // V_j and the K loaded with it consumed
        }
      }
    }
    if (elect_one()) {
      if (ok) umma_commit(&bar->o_done);
      umma_commit(&bar->fin);                     // completes once every MMA above is done
    }
    wait_phase(&bar->fin, 0, bar, a.status, false);
    __syncwarp();
    if constexpr (kSplit) {
      cluster_sync();
      cluster_sync();
    }
  } else {
    // ------------------------------------------------------------------ softmax warpgroups
    const int t = warp >> 2;                        // query tile of this warpgroup
    const int wq = warp & 3;
    const int row = wq * 32 + lane;
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    const uint32_t tS = tmem + lane_base + (uint32_t)(t * kAttnBN);
    const uint32_t tO = tmem + lane_base + kColO + (uint32_t)(t * D);
    // logit scale of this row in the log2 domain: log2(e) / sqrt(D), times 2^e_row for E4M3
    // queries (e_row in [-120, 120]: the product is exact)
    float sl2 = a.scale_log2;
    bool ok = true;
    if constexpr (kFp8) {
      // quantize this thread's query row: the bf16 row (two 64-element swizzle atoms, 16-byte
      // chunk j of row r at chunk j ^ (r & 7)) -> max |q| -> e -> E4M3 codes of q 2^-e, 128 bytes
      // in the same swizzle pattern (rows past Nq were zero-filled: e = 0, codes 0)
      if (warp_wait(&bar->q_full, 0, bar, a.status)) {
        const uint8_t* src = sQ16 + (kOne ? 0 : t) * (kAttnBM * D * 2) + row * 128;
        uint4 v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j)
          v[j] = *reinterpret_cast<const uint4*>(src + (j >> 3) * 16384 + (((j & 7) ^ (row & 7)) << 4));
        float amax = 0.0f;
#pragma unroll
        for (int j = 0; j < 16; ++j) amax = fmaxf(amax, absmax8(v[j]));
        const int e = e4m3_row_exponent(amax);
        const float inv = pow2f(-e);
        uint8_t* dst = sQ + (kOne ? 0 : t) * Lay::kQ + row * 128;
#pragma unroll
        for (int j = 0; j < 8 && (!kOne || t == 0); ++j) {
          const uint2 lo = e4m3x8(v[2 * j], inv), hi = e4m3x8(v[2 * j + 1], inv);
          *reinterpret_cast<uint4*>(dst + ((j ^ (row & 7)) << 4)) = make_uint4(lo.x, lo.y, hi.x, hi.y);
        }
        sl2 *= pow2f(e);
        // the tensor core reads shared memory through the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      } else {
        ok = false;
      }
      if (!kOne || t == 0) mbar_arrive(&bar->q8_ready);
    }
    const float2 sc2 = make_float2(sl2, sl2);
    float m = kNoMax, l = 0.0f;
    for (int it = 0; ok; ++it) {
      const int j = kOne ? 2 * it + t : it;         // kOne: this warpgroup's key set is every other tile
      if (j >= nt) break;
      if (!warp_wait(&bar->s_full[t], it & 1, bar, a.status)) { ok = false; break; }
      tc_fence_after();
      const int valid = nk - j * kAttnBN;           // keys of this tile (< 128 only in the last)
      // A tile goes in two parts, keys 0-95 and 96-127, each handed to the MMA warp as soon as
      // its P is in TMEM.  P = exp2(S*c - m) is written over S columns already read (bf16 pairs:
      // P columns 16c..16c+15 come from S columns 32c..32c+31; FP8 P V: e4m3 codes of
      // 2^6 exp2(S*c - m), four per column, P columns 8c..8c+7): the A operand of PV.  On full
      // tiles after the first, P is computed with the running max m straight away, the next
      // 32 columns' load in flight; a part whose numerators all stay within the bound is stored, else it
      // is done again by general_part.
      // general_part(Chunks<c0, kN>): chunks c0 .. c0 + kN - 1 with a max pass, and m raised when it grows by
      // more than kThr (FP8 P V: m is the running max rounded up to an integer).  O_t holds PV of
      // every key before part c0: with part 0 PV_t(j-1) is complete (see MMA order), with part 1 the
      // keys of part 0 once pva_done says so.
      // FP8 P V: tiles 1, 2, 4 .. 32 bring m up to date in every row.  m has little room before a
      // numerator leaves E4M3, most rows outgrow it early, and a raise in any one of a tile's four warps
      // delays the whole tile (480P launch 238 -> 228 us; twice as many such tiles 232)
      const bool refresh = kFp8PV && it <= 32 && (it & (it - 1)) == 0;
      auto general_part = [&](auto chunks) -> bool {
        constexpr int c0 = decltype(chunks)::first, kN = decltype(chunks)::count;
        uint32_t sv[kN][32];
#pragma unroll
        for (int c = 0; c < kN; ++c) FK_TMEM_LD32(tS + (c0 + c) * 32, sv[c]);
#pragma unroll
        for (int c = 0; c < kN; ++c) FK_TMEM_WAIT_LD32(sv[c]);
        if (valid < (c0 + kN) * 32) {                // the ragged last tile: masked keys give 0
#pragma unroll
          for (int c = 0; c < kN; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if ((c0 + c) * 32 + i >= valid) sv[c][i] = __float_as_uint(-INFINITY);
        }
        float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < kN; ++c)
#pragma unroll
          for (int i = 0; i < 32; ++i) mxa[i & 3] = fmaxf(mxa[i & 3], __uint_as_float(sv[c][i]));
        const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3]));
        const float m_new = fmaxf(m, kFp8PV ? ceilf(mx * sl2) : mx * sl2);
        const bool raise = __any_sync(0xffffffffu, m_new > m + (refresh && c0 == 0 ? 0.0f : kThr));   // warp-uniform
        float alpha = 1.0f;                          // 0 when m = kNoMax
        if (raise) {
          if constexpr (kFp8PV) {                    // integer references: an exact power of two
            const float dm = m - m_new;
            alpha = dm < -126.0f ? 0.0f : pow2f((int)dm);
          } else {
            alpha = fast_exp2(m - m_new);
          }
          l *= alpha;
          m = m_new;
        }
        const float2 nm2 = make_float2(kPShift - m, kPShift - m);
        float2 ac[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ac[i] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int c = 0; c < kN; ++c) {
          uint32_t pk[16], ov = 0;
          exp_chunk<kFp8PV>(sv[c], sc2, nm2, ac, pk, ov);
          if constexpr (kFp8PV) FK_TMEM_ST8(tS + (c0 + c) * 8, pk);
          else FK_TMEM_ST16(tS + (c0 + c) * 16, pk);
        }
        const float2 a4 = fadd2(fadd2(ac[0], ac[1]), fadd2(ac[2], ac[3]));
        l += a4.x + a4.y;
        if (raise && (it > 0 || c0 > 0)) {
          if (c0 > 0) {
            if (!warp_wait(&bar->pva_done[t], it & 1, bar, a.status)) return false;
            tc_fence_after();
          }
#pragma unroll 1
          for (int c = 0; c < D / 32; c += 2) {
            uint32_t o[32], o2[32];
            FK_TMEM_LD32(tO + c * 32, o);
            FK_TMEM_LD32(tO + c * 32 + 32, o2);
            FK_TMEM_WAIT_LD32(o);
            FK_TMEM_WAIT_LD32(o2);
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            FK_TMEM_ST32(tO + c * 32, o);
#pragma unroll
            for (int e = 0; e < 32; ++e) o2[e] = __float_as_uint(__uint_as_float(o2[e]) * alpha);
            FK_TMEM_ST32(tO + c * 32 + 32, o2);
          }
        }
        return true;
      };
      auto hand_over = [&](uint64_t* b) {            // P in TMEM -> the MMA warp
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b);
      };
      const bool direct = valid >= kAttnBN && it > 0; // uniform over the CTA
      constexpr int kW = kFp8PV ? 8 : 16;            // P words of 32 columns
      uint32_t cb[32], ov = 0;
      float2 ah[4];
      bool general = true;
      if (direct && !refresh) {
        uint32_t ca[32], pk[3 * kW];
#pragma unroll
        for (int i = 0; i < 4; ++i) ah[i] = make_float2(0.0f, 0.0f);
        const float2 nm2 = make_float2(kPShift - m, kPShift - m);
        FK_TMEM_LD32(tS, ca);
        FK_TMEM_WAIT_LD32(ca);
        FK_TMEM_LD32(tS + 32, cb);
        exp_chunk<kFp8PV>(ca, sc2, nm2, ah, pk, ov);
        FK_TMEM_WAIT_LD32(cb);
        FK_TMEM_LD32(tS + 64, ca);
        exp_chunk<kFp8PV>(cb, sc2, nm2, ah, pk + kW, ov);
        FK_TMEM_WAIT_LD32(ca);
        FK_TMEM_LD32(tS + 96, cb);
        exp_chunk<kFp8PV>(ca, sc2, nm2, ah, pk + 2 * kW, ov);
        FK_TMEM_WAIT_LD32(cb);
        general = exceeds<kFp8PV>(ah, ov);           // warp-uniform
        if (!general) {
          if constexpr (kFp8PV) {
            FK_TMEM_ST16(tS, pk);
            FK_TMEM_ST8(tS + 16, (pk + 16));
          } else {
            FK_TMEM_ST32(tS, pk);
            FK_TMEM_ST16(tS + 32, (pk + 32));
          }
          const float2 a4 = fadd2(fadd2(ah[0], ah[1]), fadd2(ah[2], ah[3]));
          l += a4.x + a4.y;
        }
      }
      if (general) {
        if (!general_part(Chunks<0, 3>{})) { ok = false; break; }
        if (direct) {                                // (not kept across the general path)
          FK_TMEM_LD32(tS + 96, cb);
          FK_TMEM_WAIT_LD32(cb);
        }
      }
      hand_over(&bar->pa_full[t]);
      general = true;
      if (direct) {
        uint32_t pk[kW];
        const float2 nm2 = make_float2(kPShift - m, kPShift - m);
#pragma unroll
        for (int i = 0; i < 4; ++i) ah[i] = make_float2(0.0f, 0.0f);
        ov = 0;
        exp_chunk<kFp8PV>(cb, sc2, nm2, ah, pk, ov);
        general = exceeds<kFp8PV>(ah, ov);
        if (!general) {
          if constexpr (kFp8PV) FK_TMEM_ST8(tS + 24, pk);
          else FK_TMEM_ST16(tS + 48, pk);
          const float2 a4 = fadd2(fadd2(ah[0], ah[1]), fadd2(ah[2], ah[3]));
          l += a4.x + a4.y;
        }
      }
      if (general && !general_part(Chunks<3, 1>{})) { ok = false; break; }
      hand_over(&bar->p_full[t]);
    }
    // ---------------------------------------------------------------- epilogue
    // every MMA is done, so the operand tiles' shared memory is free
    ok = ok && warp_wait(&bar->o_done, 0, bar, a.status);
    tc_fence_after();
    if constexpr (kSplit) {
      // Merge of the key splits: every CTA of the cluster leaves its 256 rows of unnormalised O (16-
      // byte chunk c of row g at chunk c ^ (g mod D/4): conflict-free) and their (m, l) in its shared
      // memory, and CTA r forms rows [r R, (r + 1) R) from all of them, reading whole rows of its
      // peers.  Bound by the SM-to-SM network, ~14 B per cycle and SM: 128 KB take ~9000 cycles with
      // 3 splits (17500 as 16-byte stores to the owner).
      constexpr int kRowsCta = (kOne ? 1 : 2) * kAttnBM;
      const int S = a.kv_splits, valid_rows = min(kRowsCta, a.Nq - q0), R = (valid_rows + S - 1) / S;
      float2* ml = reinterpret_cast<float2*>(smem + 2 * kAttnBM * D * 4);
      if constexpr (kOne) {
        // first the CTA's two key sets: each warpgroup forms its half of the columns of every row,
        // the other's accumulator of them through shared memory (chunk c of a row at c ^ (row mod D/8))
        constexpr int kHalf = D / 2;
        uint8_t* xo = smem + kAttnBM * D * 4 + t * (kAttnBM * kHalf * 4) + row * (kHalf * 4);
        const uint8_t* xi = smem + kAttnBM * D * 4 + (1 - t) * (kAttnBM * kHalf * 4) + row * (kHalf * 4);
        float2* mlx = ml + kAttnBM;
        const bool has = t < nt;                    // (a single key tile: the second set is empty)
        if (ok) {
#pragma unroll 1
          for (int c = 0; c < kHalf / 32; ++c) {
            uint32_t o[32];
            FK_TMEM_LD32(tO + (1 - t) * kHalf + c * 32, o);
            FK_TMEM_WAIT_LD32(o);
#pragma unroll
            for (int e = 0; e < 8; ++e)
              *reinterpret_cast<uint4*>(xo + (((c * 8 + e) ^ (row & (D / 8 - 1))) << 4)) =
                  has ? make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]) : make_uint4(0, 0, 0, 0);
          }
          mlx[t * kAttnBM + row] = make_float2(m, l);
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (ok) {
          const float2 other = mlx[(1 - t) * kAttnBM + row];
          const float M = fmaxf(m, other.x), w0 = fast_exp2(m - M), w1 = fast_exp2(other.x - M);
          uint8_t* dst = smem + row * (D * 4);
#pragma unroll 1
          for (int c = 0; c < kHalf / 32; ++c) {
            uint32_t o[32];
            FK_TMEM_LD32(tO + t * kHalf + c * 32, o);
            FK_TMEM_WAIT_LD32(o);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float4 x = *reinterpret_cast<const float4*>(xi + (((c * 8 + e) ^ (row & (D / 8 - 1))) << 4));
              float4 y = make_float4(x.x * w1, x.y * w1, x.z * w1, x.w * w1);
              if (has) {
                y.x = fmaf(__uint_as_float(o[4 * e]), w0, y.x);
                y.y = fmaf(__uint_as_float(o[4 * e + 1]), w0, y.y);
                y.z = fmaf(__uint_as_float(o[4 * e + 2]), w0, y.z);
                y.w = fmaf(__uint_as_float(o[4 * e + 3]), w0, y.w);
              }
              *reinterpret_cast<float4*>(dst + ((((t * kHalf + c * 32) / 4 + e) ^ (row & (D / 4 - 1))) << 4)) = y;
            }
          }
          if (t == 0) ml[row] = make_float2(M, l * w0 + other.y * w1);
        }
      } else if (ok) {
        const int g = t * kAttnBM + row;
        uint8_t* dst = smem + g * (D * 4);
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          FK_TMEM_LD32(tO + c * 32, o);
          FK_TMEM_WAIT_LD32(o);
#pragma unroll
          for (int e = 0; e < 8; ++e)
            *reinterpret_cast<uint4*>(dst + (((c * 8 + e) ^ (g & (D / 4 - 1))) << 4)) =
                make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
        }
        ml[g] = make_float2(m, l);
      }
      cluster_sync();                               // every CTA's rows are in place
      const int rows = min(R, valid_rows - split * R);
      bf16* orow = a.O + ((int64_t)(q0 + split * R) * a.H + head) * D;
      if (S <= 2) merge_rows<D, 2, 2>(su32(smem), su32(ml), S, split * R, rows, orow, a.H * D, warp, lane);
      else if (S <= 4) merge_rows<D, 4, 1>(su32(smem), su32(ml), S, split * R, rows, orow, a.H * D, warp, lane);
      else merge_rows<D, 8, 1>(su32(smem), su32(ml), S, split * R, rows, orow, a.H * D, warp, lane);
      cluster_sync();                               // every peer has read this CTA's rows
    } else if (ok) {
      // normalise, and through the warp's own 32 rows of shared memory (16-byte chunk c of row r at
      // chunk c ^ (r mod D/8)) to whole rows of O: a thread storing its own row took ~3 us per CTA
      const float inv = 1.0f / l;
      uint8_t* stage = smem + warp * (32 * D * 2);
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t o[32];
        FK_TMEM_LD32(tO + c * 32, o);
        FK_TMEM_WAIT_LD32(o);
#pragma unroll
        for (int e = 0; e < 32; e += 8) {
          uint4 v;
          v.x = pack_bf16(__uint_as_float(o[e + 0]) * inv, __uint_as_float(o[e + 1]) * inv);
          v.y = pack_bf16(__uint_as_float(o[e + 2]) * inv, __uint_as_float(o[e + 3]) * inv);
          v.z = pack_bf16(__uint_as_float(o[e + 4]) * inv, __uint_as_float(o[e + 5]) * inv);
          v.w = pack_bf16(__uint_as_float(o[e + 6]) * inv, __uint_as_float(o[e + 7]) * inv);
          *reinterpret_cast<uint4*>(stage + lane * (D * 2) + (((c * 4 + e / 8) ^ (lane & (D / 8 - 1))) << 4)) = v;
        }
      }
      __syncwarp();
      constexpr int kLanes = D / 8;                 // lanes of one row
      const int cl = lane % kLanes;
#pragma unroll
      for (int r0 = 0; r0 < 32; r0 += 32 / kLanes) {
        const int r = r0 + lane / kLanes, q = q0 + t * kAttnBM + wq * 32 + r;
        const uint4 v = *reinterpret_cast<const uint4*>(stage + r * (D * 2) + ((cl ^ (r & (D / 8 - 1))) << 4));
        if (q < a.Nq) *reinterpret_cast<uint4*>(a.O + ((int64_t)q * a.H + head) * D + cl * 8) = v;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem),
                 "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------
// Offline head profiling (Sec. 4.1, Eq. 1): per head, the attention mass that the queries of
// the generated chunk put on the generated chunk, the transition (anchor) frame and the sink
// frames, out of a full softmax over every key of the attention window.  Keys are ordered
// [generated | sink | other history | transition].  S = Q K^T runs on the tensor cores
// (tcgen05, S double-buffered in 256 TMEM columns); no P V product is needed.  Per row the
// softmax statistics are kept online (running max, total sum, and the three class sums,
// rescaled together); the per-row fractions are summed per head in double.  A cluster of k >= 2
// CTAs handles one (head, 128-row query tile), each CTA a k-th of the key tiles (two fill the SMs
// in about three even waves at 480P instead of two, the second half empty; small windows take
// more, see launch_head_profile); the other CTAs write their row statistics into the first's shared
// memory (distributed shared memory, between two cluster barriers), and the first merges the ranges.
// What bounds it: the statistics warps (the exponentials of a tile alone hold an SM sub-partition's
// special-function unit for 512 cycles, as long as the MMAs take; each is active 63% of the time).
// With one set of statistics warps per CTA the two CTAs of an SM fell into step, computing and
// waiting at the same time.  12 heads, 4680 queries, 34320 keys, launches back to back: 372 us (405 with one
// set, its loads not overlapped and a branch per key in tiles of two classes; D = 64 320, was 389), 351-402 by
// box for a launch on a flushed L2; 8 heads, 534
// queries, 1246 keys, D = 64: 10.4 us (16.4 with two CTAs per query tile).  Tried: S released before
// the sums (registers for 128 columns), no faster; loads running ahead into the next tile, slower; the
// query tile in tensor memory, which halves the operand fetch from shared memory (8 KB in the 64
// cycles of a 128x128x16 MMA), no faster.
//   warps 0-7  statistics of rows 0..127 (TMEM lanes), one thread per row, warps 0-3 on the even key
//              tiles, 4-7 on the odd ones (merged at the end);
//   warp 8     TMA: the query tile once, key tiles into a two-stage ring;
//   warp 9     tcgen05.mma: S_b = Q K_j^T for b = j mod 2, once the statistics warps have
//              read S_b of tile j - 2.
constexpr int kProfThreads = 320;
constexpr int kWarpProfTma = 8;                    // warps 0-3 / 4-7: statistics of even / odd key tiles
constexpr int kWarpProfMma = 9;

template <int D>
struct ProfLayout {
  static constexpr int kQ = kAttnBM * D * 2;
  static constexpr int kK = kAttnBN * D * 2;
  static constexpr int kOffQ = 0;
  static constexpr int kOffK = kOffQ + kQ;
  static constexpr int kOffBar = kOffK + 2 * kK;
  static constexpr int kOffOdd = kOffBar + 256;       // row statistics of the odd key tiles
  static constexpr int kOffPart = kOffOdd + kAttnBM * 8 * 4;   // row statistics of peer 1 of the cluster
  static constexpr int kSmem = kOffPart + kAttnBM * 8 * 4 + 1024;   // + alignment slack; two CTAs per SM
  static_assert((kMaxKvSplits - 2) * kAttnBM * 8 * 4 <= 2 * kK, "statistics of peers 2.. over the key stages");
};

template <int D>
__global__ void __launch_bounds__(kProfThreads, 2)
profile_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
               const ProfArgs a) {
  using Lay = ProfLayout<D>;
  constexpr int kHalves = D / 64;
  constexpr uint32_t kTmemCols = 256;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* sQ = smem + Lay::kOffQ;
  uint8_t* sK = smem + Lay::kOffK;
  AttnBarriers* bar = reinterpret_cast<AttnBarriers*>(smem + Lay::kOffBar);
  // barrier use: q_full, k_full/k_empty (key ring), s_full[b] (S_b written), p_full[b]
  // (S_b read by the four statistics warps), fin

  // [row][8]: m l cg cs ct ok of CTA r >= 1 of the cluster; of the third CTA on over the key
  // stages, once every CTA is done with them
  auto part_of = [&](uint32_t r) {
    return reinterpret_cast<float*>(r == 1 ? smem + Lay::kOffPart : sK + (r - 2) * (kAttnBM * 8 * 4));
  };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (warp & 3) * 32 + lane;           // query row of a statistics thread
  const int grp = warp >> 2;                        // its key tiles: even (0) or odd (1)
  // A cluster of k CTAs = one (head, query tile); CTA r of the cluster takes key tiles [j0, j0 + nt)
  // of the head's window, the r-th of k even ranges.
  uint32_t rank, k;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(k));
  const int pair = blockIdx.x / k;
  const int head = pair / a.n_qtiles;
  const int q0 = (pair - head * a.n_qtiles) * kAttnBM;
  const int nk = a.Nk;
  const int nt_all = (nk + kAttnBN - 1) / kAttnBN;
  const int j0 = (int)((int64_t)nt_all * rank / k);
  const int nt = (int)((int64_t)nt_all * (rank + 1) / k) - j0;   // may be 0 (fewer key tiles than CTAs)
  // row statistics of this CTA's keys (statistics warps): running max (log2 domain), total
  // sum and the class sums, all relative to m
  float m = kNoMax, l = 0.0f, cg = 0.0f, cs = 0.0f, ct = 0.0f;
  bool ok = true;

  // the TMA warp makes the barriers and starts the first loads before the CTA meets
  auto load_k = [&](int j) {                          // key tile j into its stage
    const int st = j & 1;
    mbar_expect_tx(&bar->k_full[st], Lay::kK);
    for (int h = 0; h < kHalves; ++h)
      tma_load_3d(sK + st * Lay::kK + h * 16384, &tmK, &bar->k_full[st], h * 64, head, (j0 + j) * kAttnBN);
  };
  if (warp == kWarpProfTma && lane == 0) {
    mbar_init(&bar->q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar->k_full[i], 1);
      mbar_init(&bar->k_empty[i], 1);
      mbar_init(&bar->s_full[i], 1);
      mbar_init(&bar->p_full[i], 4);
    }
    mbar_init(&bar->fin, 1);
    bar->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&bar->q_full, Lay::kQ);
    for (int h = 0; h < kHalves; ++h)
      tma_load_3d(sQ + h * 16384, &tmQ, &bar->q_full, h * 64, head, q0);
    for (int j = 0; j < min(2, nt); ++j) load_k(j);
  }
  __syncwarp();
  if (warp == kWarpProfMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(su32(&bar->tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  if (k == 2) cluster_arrive();                     // this CTA has started (waited for before the remote stores)

  if (warp == kWarpProfTma) {
    if (lane == 0) {
      int lastK[2] = {nt > 0 ? 0 : -1, nt > 1 ? 0 : -1};
      bool ok = true;
      for (int j = 2; j < nt; ++j) {
        const int st = j & 1, u = j >> 1;
        if (!wait_phase(&bar->k_empty[st], (u - 1) & 1, bar, a.status)) { ok = false; break; }
        load_k(j);
        lastK[st] = u;
      }
      if (!ok) {   // drain every load this thread issued before the CTA exits
        wait_phase(&bar->q_full, 0, bar, a.status, false);
        for (int st = 0; st < 2; ++st)
          if (lastK[st] >= 0) wait_phase(&bar->k_full[st], lastK[st] & 1, bar, a.status, false);
      }
    }
    __syncwarp();
  } else if (warp == kWarpProfMma) {
    constexpr uint32_t kIdQK = idesc_bf16(kAttnBM, kAttnBN, 0);
    const uint64_t dQ = sdesc(su32(sQ), 16, 1024), dK = sdesc(su32(sK), 16, 1024);
    bool ok = warp_wait(&bar->q_full, 0, bar, a.status);
    for (int j = 0; j < nt && ok; ++j) {
      const int st = j & 1, u = j >> 1;
      if (!warp_wait(&bar->k_full[st], u & 1, bar, a.status) ||
          (j >= 2 && !warp_wait(&bar->p_full[st], (u - 1) & 1, bar, a.status))) { ok = false; break; }
      tc_fence_after();
      if (elect_one()) {
        const uint64_t db = dK + (uint32_t)(st * (Lay::kK >> 4));
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (uint32_t)((kk >> 2) * 1024 + (kk & 3) * 2);
          umma(tmem + (uint32_t)(st * kAttnBN), dQ + off, db + off, kIdQK, kk > 0 ? 1u : 0u);
        }
        umma_commit(&bar->s_full[st]);
        umma_commit(&bar->k_empty[st]);
      }
    }
    if (elect_one()) umma_commit(&bar->fin);      // completes once every MMA above is done
    wait_phase(&bar->fin, 0, bar, a.status, false);
    __syncwarp();
  } else {
    const uint32_t tS = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(grp * kAttnBN);
    const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
    // key classes are contiguous ranges in the order generated, sink, other, transition
    auto key_class = [&](int key) { return key < a.g_end ? 0 : key < a.s_end ? 1 : key >= a.t_begin ? 3 : 2; };
    auto add = [&](int cls, float sum) {
      l += sum;
      if (cls == 0) cg += sum;
      else if (cls == 1) cs += sum;
      else if (cls == 3) ct += sum;
    };
    for (int j = grp; j < nt; j += 2) {              // S_j is in buffer j mod 2
      if (!warp_wait(&bar->s_full[grp], (j >> 1) & 1, bar, a.status)) { ok = false; break; }
      tc_fence_after();
      auto release = [&] {                           // S has been read
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar->p_full[grp]);
      };
      // A full tile of one key class after the first (every row then has a finite running max m):
      // the exponentials with m straight away, the next 32 columns' load in flight.  The tile's sum
      // bounds each term, so only a sum above 2^8 (128 keys: some key at least 1 above m in log2
      // units) needs the general path, which does the tile again.
      const int k0 = (j0 + j) * kAttnBN;
      if (j > 1 && nk - k0 >= kAttnBN && key_class(k0) == key_class(k0 + kAttnBN - 1)) {   // CTA-uniform
        const float2 nm2 = make_float2(-m, -m);
        float2 a2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a2[i] = make_float2(0.0f, 0.0f);
        uint32_t va[32], vb[32];
        FK_TMEM_LD32(tS, va);
        FK_TMEM_WAIT_LD32(va);
        FK_TMEM_LD32(tS + 32, vb);
        exp_sum(va, sc2, nm2, a2);
        FK_TMEM_WAIT_LD32(vb);
        FK_TMEM_LD32(tS + 64, va);
        exp_sum(vb, sc2, nm2, a2);
        FK_TMEM_WAIT_LD32(va);
        FK_TMEM_LD32(tS + 96, vb);
        exp_sum(va, sc2, nm2, a2);
        FK_TMEM_WAIT_LD32(vb);
        exp_sum(vb, sc2, nm2, a2);
        const float2 s2 = fadd2(fadd2(a2[0], a2[1]), fadd2(a2[2], a2[3]));
        const float sum = s2.x + s2.y;
        if (!__any_sync(0xffffffffu, sum > 256.0f)) {                    // warp-uniform
          release();
          add(key_class(k0), sum);
          continue;
        }
      }
      // General path: 32 columns at a time, with a max pass; classes by selection (a branch per key
      // took 12000 cycles for a tile of two classes)
#pragma unroll 1
      for (int c0 = 0; c0 < 4; ++c0) {
        const int kb = k0 + c0 * 32;                 // first key of these columns
        const int valid = min(32, nk - kb);          // uniform over the CTA
        float sv[32];
        {
          uint32_t u[32];
          FK_TMEM_LD32(tS + c0 * 32, u);
          FK_TMEM_WAIT_LD32(u);
#pragma unroll
          for (int c = 0; c < 32; ++c) sv[c] = c < valid ? __uint_as_float(u[c]) : -INFINITY;
        }
        if (c0 == 3) release();
        if (valid <= 0) continue;
        float mxa[4];                                // four independent max chains
#pragma unroll
        for (int i = 0; i < 4; ++i) mxa[i] = sv[i];
#pragma unroll
        for (int c = 4; c < 32; ++c) mxa[c & 3] = fmaxf(mxa[c & 3], sv[c]);
        const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3]));
        const float m_new = fmaxf(m, mx * a.scale_log2);
        if (__any_sync(0xffffffffu, m_new > m + kRescaleThreshold)) {   // warp-uniform
          const float alpha = fast_exp2(m - m_new);  // 0 when m = kNoMax
          l *= alpha;
          cg *= alpha;
          cs *= alpha;
          ct *= alpha;
          m = m_new;
        }
        float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          sv[c] = fast_exp2(fmaf(sv[c], a.scale_log2, -m));
          sum[c & 3] += sv[c];
        }
        const float all = (sum[0] + sum[1]) + (sum[2] + sum[3]);
        const int cls_first = key_class(kb), cls_last = key_class(kb + valid - 1);
        if (cls_first == cls_last) {
          add(cls_first, all);
        } else {
          const int ng = a.g_end - kb, ns = a.s_end - kb, nt0 = a.t_begin - kb;
          float pg[2] = {0.0f, 0.0f}, ps[2] = {0.0f, 0.0f}, pt[2] = {0.0f, 0.0f};
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            pg[c & 1] = fmaf(c < ng ? 1.0f : 0.0f, sv[c], pg[c & 1]);
            ps[c & 1] = fmaf(c >= ng && c < ns ? 1.0f : 0.0f, sv[c], ps[c & 1]);
            pt[c & 1] = fmaf(c >= nt0 ? 1.0f : 0.0f, sv[c], pt[c & 1]);
          }
          l += all;
          cg += pg[0] + pg[1];
          cs += ps[0] + ps[1];
          ct += pt[0] + pt[1];
        }
      }
    }
  }
  // merge of a row's statistics with those of other keys: with M = max(m0, m1), every sum
  // s = s0 2^(m0 - M) + s1 2^(m1 - M)
  auto merge = [&](const float* pp) {
    const float pm = pp[0];
    ok = ok && pp[5] != 0.0f;                       // warp-uniform: one warp writes a row block
    const float M = fmaxf(m, pm);
    const float w0 = fast_exp2(m - M), w1 = fast_exp2(pm - M);   // 0 where no key had a finite logit
    m = M;
    l = l * w0 + pp[1] * w1;
    cg = cg * w0 + pp[2] * w1;
    cs = cs * w0 + pp[3] * w1;
    ct = ct * w0 + pp[4] * w1;
  };
  if (warp < kWarpProfTma) {                        // the odd tiles' statistics to the even tiles' threads
    float* odd = reinterpret_cast<float*>(smem + Lay::kOffOdd) + row * 8;
    if (grp == 1) {
      *reinterpret_cast<float4*>(odd) = make_float4(m, l, cg, cs);
      *reinterpret_cast<float2*>(odd + 4) = make_float2(ct, ok ? 1.0f : 0.0f);
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (grp == 0) merge(odd);
  }
  // Distributed shared memory may be written only once the owner has started, and the key stages (k > 2)
  // only once it is done with them.  With two CTAs the barrier was arrived at when each began, so that
  // neither waits here for the other's key range.
  if (k == 2) cluster_wait();
  else cluster_sync();
  if (warp < 4) {
    if (rank > 0) {
      // this CTA's row statistics go to its slot of the same row in the first CTA's shared memory
      const uint32_t dst = map_peer(su32(part_of(rank) + row * 8), 0);
      asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(dst), "f"(m), "f"(l),
                   "f"(cg), "f"(cs) : "memory");
      asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" :: "r"(dst + 16u), "f"(ct),
                   "f"(ok ? 1.0f : 0.0f) : "memory");
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kWarpProfMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem),
                 "r"(kTmemCols) : "memory");
  }
  // every thread of the cluster: the other CTAs' statistics have landed
  cluster_sync();
  if (rank == 0 && warp < 4) {
    for (uint32_t r = 1; r < k; ++r) merge(part_of(r) + row * 8);
    if (ok) {
      const bool in = q0 + row < a.Nq;
      float fg = in ? cg / l : 0.0f, fs = in ? cs / l : 0.0f, ft = in ? ct / l : 0.0f;
      float rows = in ? 1.0f : 0.0f;
#pragma unroll
      for (int sft = 16; sft >= 1; sft >>= 1) {
        fg += __shfl_xor_sync(0xffffffffu, fg, sft);
        fs += __shfl_xor_sync(0xffffffffu, fs, sft);
        ft += __shfl_xor_sync(0xffffffffu, ft, sft);
        rows += __shfl_xor_sync(0xffffffffu, rows, sft);
      }
      if (lane == 0 && rows > 0.0f) {
        double* mh = a.mass + (int64_t)head * 4;
        atomicAdd(mh + 0, (double)rows);
        atomicAdd(mh + 1, (double)fg);
        atomicAdd(mh + 2, (double)ft);
        atomicAdd(mh + 3, (double)fs);
      }
    }
  }
}

}  // namespace

cudaError_t launch_head_profile(int head_dim, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                                const ProfArgs& a, cudaStream_t s) {
  // Key ranges per (head, query tile): two, or more while the CTAs (two per SM) all run at once.
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)a.n_qtiles * a.H;
  const int key_tiles = (a.Nk + kAttnBN - 1) / kAttnBN;
  int k = 2;
  while (k < kMaxKvSplits && tiles * (k + 1) <= 2 * sms * 9 / 10 && k + 1 <= key_tiles) ++k;
  void (*kern)(const CUtensorMap, const CUtensorMap, const ProfArgs) =
      head_dim == 128 ? profile_kernel<128> : profile_kernel<64>;
  const int smem = head_dim == 128 ? ProfLayout<128>::kSmem : ProfLayout<64>::kSmem;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * k));
  cfg.blockDim = dim3(kProfThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)k;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, tmQ, tmK, a);
}

namespace {
using AttnKern = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const AttnArgs);
// kernels of one head_dim and precision: [0] no key splits, [1] key splits, [2] one query tile per CTA
struct AttnKerns {
  AttnKern k[3];
  int smem;
};
template <int D, bool kFp8, bool kFp8PV>
AttnKerns attn_kernels() {
  return {{attn_kernel<D, false, kFp8, kFp8PV>, attn_kernel<D, true, kFp8, kFp8PV>,
           attn_kernel<D, true, kFp8, kFp8PV, true>},
          Layout<D, kFp8, kFp8PV>::kSmem};
}
AttnKerns attention_kernels(int head_dim, int precision) {
  if (head_dim == 64) return attn_kernels<64, false, false>();
  if (precision == FK_ATTN_FP8) return attn_kernels<128, true, true>();
  if (precision == FK_ATTN_FP8_QK) return attn_kernels<128, true, false>();
  return attn_kernels<128, false, false>();
}
// launch configuration with programmatic dependent launch and, for key splits, a cluster of them
void attention_config(int splits, int grid, int smem, cudaStream_t s, cudaLaunchConfig_t* cfg,
                      cudaLaunchAttribute* attr) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)grid);
  cfg->blockDim = dim3(kAttnThreads);
  cfg->dynamicSmemBytes = (size_t)smem;
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)splits;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = splits > 1 ? 2 : 1;
}
}  // namespace

cudaError_t attention_prepare(int head_dim) {
  for (int precision : {FK_ATTN_BF16, FK_ATTN_FP8_QK, FK_ATTN_FP8}) {
    const AttnKerns ks = attention_kernels(head_dim, precision);
    for (AttnKern kern : ks.k) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ks.smem);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t attention_clusters(int head_dim, int precision, int splits, int* n) {
  const AttnKerns ks = attention_kernels(head_dim, precision);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  attention_config(splits, splits, ks.smem, nullptr, &cfg, attr);
  return cudaOccupancyMaxActiveClusters(n, ks.k[1], &cfg);
}

void launch_attention(int head_dim, int precision, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                      const CUtensorMap& tmV, const AttnArgs& a, cudaStream_t s) {
  const AttnKerns ks = attention_kernels(head_dim, precision);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  attention_config(a.kv_splits, a.n_qtiles * a.H * a.kv_splits, ks.smem, s, &cfg, attr);
  cudaLaunchKernelEx(&cfg, ks.k[a.one_qtile ? 2 : a.kv_splits > 1 ? 1 : 0], tmQ, tmK, tmV, a);
}

}  // namespace fk
