// LR-reconstructed attention for the new tokens of a turn on the 5th-generation tensor cores.
//
// One thread block = up to 128 query rows of one kv head (row = new token i * G + head-in-group) against
// the whole visible context, 128 tokens per step:
//   S  = Q K_base^T + Q~ L_K^T                 tcgen05.mma, A/B from shared memory, S in TMEM (2 buffers)
//   P  = exp2(S*scale - m)                     two softmax warpgroups, one thread per TMEM lane (= query row);
//                                              packed bf16 in its own 64 TMEM columns
//   O' += P [V_base | L_V]                      tcgen05.mma with A = P from TMEM; O' in TMEM holds the numerator
//                                              (hd columns) and U = P L_V (r_v columns)
// and finally out = (O + s_v U B_v) / l.  Both folds are MMAs too: Q~ = s_k Q B_k^T before the first step (product in the
// first columns of S buffer 0, scaled and rounded to bf16 by the softmax threads), and O += (s_v U) B_v after the
// last (s_v U enters as three bf16 terms, i.e. with all 24 bits of its fp32 value).  The caches arrive by TMA into
// rings of stages guarded by mbarriers: one box per page and 64-column slab when a block table scatters the pages,
// one box per slab for the whole 128-token stage (4-D tensor map) when the pages are consecutive; the query tile and
// the two B slices are TMA boxes as well.
//
// TMEM columns: S0 [0,128) | S1 [128,256) | P, one or two buffers of 64 | O', hd + r_v <= 192.  Because P does not
// overlay S, an S buffer is free as soon as the softmax threads have pulled it into registers, so
// Q K^T runs two steps ahead of the softmax.  P has two buffers where O' leaves room for them (hd + r_v <= 128) and
// is rewritten once the P V' that read the buffer has retired.
//
// Softmax.  A step costs the special-function unit about 1000 cycles, and a warp's own chain (scores out of TMEM,
// maximum, exponentials, P into TMEM, barriers) adds about as many cycles of latency in which it issues none.  So the two
// warpgroups take alternate steps: each has two steps' time for one chain, and one's exponentials run under the other's
// latencies.  A thread owns a whole row of a step (128 scores in registers), so no maximum is exchanged between threads;
// what the warpgroups hand to each other is the row's reference maximum, one word through shared memory behind a
// named barrier per warp pair, decided right after a step's scores are in registers.  The reference is raised
// only when the maximum grows by more than 8 (log2 domain), so O' is rescaled a handful of times per row instead of
// at every step; P stays below 2^8.  The denominator: for 0 < r_v < 64 the rounded weights that the MMA sees are summed, by the
// MMA: behind each k step of P V' a second one of N = 16 multiplies the same P with a constant tile of ones (512 bytes of
// shared memory, sixteen equal columns behind O').  The softmax threads are left with four instructions per pair of
// scores instead of seven (8192 over 24576: 4147 -> 3895 us; 512 over 32768 with both projections: 316 -> 297).  Otherwise, in the work-list
// form (which would spill) and in most split-context forms at head_dim 128, they sum in fp32, two values per instruction.  (Unrounded, the sum left a
// row dominated by one token up to 2^-8 off, on top of its own rounding, and the error against float64 5 .. 15 % higher
// where a few tokens carry a row.)  Measured for the same sum and slower: a column of ones beside L_V in the value stage -
// written into every landed stage by the issuing warp it takes 600 cycles of a step, by the softmax threads 6 % more time on
// the mean -, the ones behind all eight k steps instead of between them (330 against 272 us), a warp-level mma.sync
// against a selection matrix, which competes with tcgen05, and adds of fp32 and bf16 (turn of 512: 6 % slower).
//
// Warp roles: warp 0 = TMA producer of the key ring, warp 3 = TMA producer of the value ring
// (keys are released right after S is computed, values only after O' is updated, so the two rings run
// at different distances ahead), warp 1 = TMEM owner + Q K^T issuer, warp 2 = P V' issuer (an MMA costs
// its issuing thread about a hundred cycles, so the two streams are issued by different threads), warps 4-11 = softmax
// / correction / epilogue, warps 12-15 = more TMA issuers for paged caches: a copy costs its issuing warp about a hundred
// cycles, and a step of a paged cache is up to 48 copies (two slabs and the LR rows of eight pages, keys and values), so
// each warp takes eight of them (two issuers: 2250 cycles per step at head_dim 128; six: 1750, bound by the softmax).
// Registers are re-split at kernel start: 216 per softmax thread, 40 for the other eight warps
// (8 x 216 + 8 x 40 = 16 x 128).  Nothing may spill in the step loop: shared memory is addressed in its own address space
// (a base rounded up as an integer made every access a generic one with a 64-bit address: 5 % of the time of a turn), and the
// work-list form reads its piece's data again for the epilogue.  Every mbarrier wait is bounded and falls through with PRECC_STATUS_TIMEOUT.
//
// Two more instantiations of the same kernel.  VH: the value ring holds units of 64 tokens instead of whole
// steps (where one value stage fits beside two key stages but two do not), a unit being freed as soon as its
// four k-steps of P V' retire.  WL: the work-list launch - a 1-D grid in which the first (row tiles x kv heads)
// blocks stop `helper_p` steps into their tile and the remaining blocks share the tails of all tiles, several
// pieces each with the block drained in between; the pieces of a tile meet through fp32 records in a
// caller-provided workspace, and the block that arrives last at the tile's ticket merges them in piece order.
#pragma once
#include <type_traits>

#include "prefill_plan.h"
#include "tc_common.cuh"

namespace precc {

// Tensor maps of one launch: caches, query rows, and the agent's B slices.
struct PrefillTcMaps { CUtensorMap k, v, lk, lv, q, bk, bv; };

struct PrefillTcParams {
  __nv_bfloat16* out;
  const int32_t* block_table;
  uint32_t* status;
  int64_t n_blocks;
  int S, T, first_block;
  int n_q, n_kv, group;
  int tok_per_tile;            // 128 / group
  int k_stages, v_stages;      // depth of the key ring and of the value ring
  int v_half;                  // 1: the value ring holds v_stages units of 64 tokens (half a step) instead of whole steps - where
                               //    shared memory has room for one and a half value stages but not for two
  int contig;                  // 1: no block table; the tensor maps fetch a whole 128-token stage per box
  int k_logical;               // 1: the key map covers a scratch copy of this sequence's keys in logical block order (whole-stage boxes
                               //    from block 0), whatever the layout of the value side
  int longest_first;           // 1: block x = 0 takes the LAST row tile (longest causal reach), so the tail of the grid is short blocks
  float scale_log2, s_k, s_v;
  unsigned long long* trace;   // PRECC_PF_TRACE builds only: [steps][16] clock stamps of block (0, 0)
  // Work-list launch (helper_p > 0; 1-D grid of tiles + n_helpers blocks, no cluster): block b < tiles takes steps
  // [0, helper_p) of tile b, the n_helpers blocks behind them share the tails of all tiles; the pieces of a tile meet
  // through records in `ws_rec`, and the block that arrives last at the tile's ticket merges them.
  int helper_p, n_helpers, row_tiles;
  float* ws_rec;               // [2 * tiles + n_helpers][PrefillTcCfg::REC_FLOATS]
  unsigned int* ws_ticket;     // [tiles], zero before the launch and again after it
};

// Timeline stamps for tuning (compiled in with -DPRECC_PF_TRACE; slot meanings at the call sites).
#ifdef PRECC_PF_TRACE
#define PTC_STAMP(p, j, slot)                                                                    \
  do {                                                                                           \
    if ((p).trace && blockIdx.x == 0 && blockIdx.y == 0 && (j) < 64) (p).trace[(j) * 16 + (slot)] = clock64(); \
  } while (0)
// work-list launch: wall-clock stamps of every block's pieces (thread 0 of the softmax warps), behind the step stamps
#define PTC_WL_STAMP(p, seg, slot)                                                               \
  do {                                                                                           \
    if ((p).trace && (p).helper_p > 0 && threadIdx.x == PTC_FIRST_SM_WARP * 32 && (seg) < 16) {   \
      unsigned long long t__;                                                                    \
      asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t__));                                 \
      (p).trace[1024 + blockIdx.x * 128 + (seg) * 8 + (slot)] = t__;                             \
    }                                                                                            \
  } while (0)
#else
#define PTC_STAMP(p, j, slot) do { } while (0)
#define PTC_WL_STAMP(p, seg, slot) do { } while (0)
#endif

constexpr int PTC_FIRST_SM_WARP = 4;                 // warps 0..3: key producer, Q K^T issuer, P V' issuer, value producer
constexpr int PTC_SOFTMAX_WARPS = 8;                 // two warpgroups, taking alternate steps
constexpr int PTC_FIRST_HELPER = PTC_FIRST_SM_WARP + PTC_SOFTMAX_WARPS;   // four more TMA issuers (paged caches)
constexpr int PTC_THREADS = (PTC_FIRST_HELPER + 4) * 32;
constexpr int PTC_SM_REGS = 216, PTC_CTL_REGS = 40;  // 256 x 216 + 256 x 40 = 512 x 128, the launch's registers
constexpr int PTC_SMEM_LIMIT = 232448;   // dynamic shared memory a block can opt into on this architecture
constexpr int PTC_FIXED_BARS = 13; // barriers besides the two per ring stage
constexpr int PTC_XCH_BYTES = 4 * 512;   // [2][128] reference maxima | [2][128] partial denominators or the tile of ones
constexpr float PTC_RAISE = 8.f;  // the running maximum is raised only when it grows by more than this
constexpr int PTC_MAX_SPLIT = 8;  // blocks of a split-context cluster at most
constexpr int PTC_TAB_BYTES = (2 * PTC_MAX_XT + 8 + 4 * PTC_MAX_SEG) * 4;   // tail lengths | their prefix sums | scalars | piece list

template <int HD, int RK, int RV>
struct PrefillTcCfg {
  static constexpr int SLABS = HD / 64;                      // 64-column slabs of a base row
  static constexpr int SLAB_BYTES = PTC_TOK * 128;            // 128 rows x 128 bytes
  static constexpr int Q_BYTES = SLABS * SLAB_BYTES;
  static constexpr int RKP = RK == 8 ? 16 : RK;               // rank 8 rides as a zero-padded k step of 16
  static constexpr int QX_BYTES = RK > 0 ? PTC_TOK * RKP * 2 : 0;
  static constexpr int KV_BYTES = SLABS * SLAB_BYTES;
  static constexpr int LK_BYTES = PTC_TOK * RKP * 2;
  static constexpr int LV_BYTES = PTC_TOK * RV * 2;
  static constexpr int KSTAGE = KV_BYTES + LK_BYTES;          // {K_base slabs | L_K} of 128 tokens
  static constexpr int VSLABS = SLABS + (RV > 0 ? 1 : 0);     // L_V rides as one more 64-column slab (zero padded)
  static constexpr int RVP = RV == 8 ? 16 : RV;               // value-side coordinates as the MMAs see them (rank 8: zero-padded)
  static constexpr int OW = HD + RVP;                         // columns of O' in TMEM: [O | U]
  // The denominator is the sum of the bf16 weights that the P V' MMA multiplies, so that the rounding of a dominant weight
  // cancels; with no value adapter or rank 64 (no tensor memory left beside O') it is the sum of the unrounded ones.
  static constexpr bool L_ROUNDED = RV > 0 && RV < 64;
  static constexpr int OWL = OW + (L_ROUNDED ? 16 : 0);       // and, where the MMA sums the denominator, sixteen copies of it
  static constexpr int VSTAGE = VSLABS * SLAB_BYTES;          // {V_base slabs | L_V slab}
  static constexpr int K_PAGE_TX = PAGE * (HD + RKP) * 2;      // bytes one page contributes to a key stage
  static constexpr int V_PAGE_TX = PAGE * VSLABS * 128;
  static constexpr int UPW = RVP / 2;                         // TMEM columns of one bf16 term of s_v U
  static constexpr int BV_BYTES = RVP * HD * 2;               // the B_v slice, one more item of the key ring behind the last step
  static constexpr int SPLIT_XS = HD + 4;                     // row stride (floats) of a partial: the adapter term is added before partials are merged
  // split-context merge area (laid over the Q tile, the folded-query tile and the rings): partial rows [O | m | l | - | -], then
  // the peers' partials of the rows this block finishes (at most 6 x 19 rows, clusters of seven)
  static constexpr int SPLIT_BYTES = (128 + 114) * SPLIT_XS * 4;
  static constexpr int REC_FLOATS = 128 * SPLIT_XS + 256;     // a tile's partial in global memory: O rows | m[128] | l[128]
  static constexpr int PB = OW <= 128 ? 2 : 1;                // P buffers
  static constexpr int TMEM_P = 2 * PTC_TOK;                  // packed bf16 P (64 columns each) after the two S buffers
  static constexpr int TMEM_O = TMEM_P + PB * (PTC_TOK / 2);  // O': at most 320 + 192 or 384 + 128 = 512
  static_assert(TMEM_O + OWL <= 512, "tensor memory");
  __host__ __device__ static constexpr int smem_bytes(int ks, int vs, bool v_half = false) { return Q_BYTES + QX_BYTES + ks * KSTAGE + vs * (v_half ? VSTAGE / 2 : VSTAGE) + 320 + PTC_XCH_BYTES + PTC_TAB_BYTES + 1024; }
  // one whole value stage fits beside two key stages, two do not, three half-step units do (head_dim 128 with rank 64)
  static constexpr bool V_HALF_CAPABLE = smem_bytes(2, 2) > PTC_SMEM_LIMIT && smem_bytes(2, 1) <= PTC_SMEM_LIMIT && smem_bytes(2, 3, true) <= PTC_SMEM_LIMIT;
  static constexpr bool supported = (HD == 64 || HD == 128) && (RK == 0 || RK == 8 || RK == 16 || RK == 32 || RK == 64) &&
                                    (RV == 0 || RV == 8 || RV == 16 || RV == 32 || RV == 64);
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar) : "memory");
}

// layout_type field of a shared-memory matrix descriptor for rows of `row_bytes`
__device__ __forceinline__ constexpr uint64_t umma_layout_for(int row_bytes) {
  return row_bytes >= 128 ? 2ull : (row_bytes == 64 ? 4ull : 6ull);
}
// K-major operand: rows of `row_bytes` (one swizzle span), 8-row groups `8*row_bytes` apart.
__device__ __forceinline__ uint64_t umma_desc_kmajor(uint32_t saddr, int row_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFF) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>((8 * row_bytes) >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= umma_layout_for(row_bytes) << 61;
  return d;
}
// MN-major operand (rows = k index, `row_bytes` of contiguous MN elements per row): 8-row groups
// `8*row_bytes` apart (stride offset), successive MN blocks `mn_block_stride` bytes apart (leading offset).
__device__ __forceinline__ uint64_t umma_desc_mnmajor(uint32_t saddr, int row_bytes, int mn_block_stride) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFF) >> 4);
  d |= static_cast<uint64_t>((mn_block_stride >> 4) & 0x3FFF) << 16;
  d |= static_cast<uint64_t>((8 * row_bytes) >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= umma_layout_for(row_bytes) << 61;
  return d;
}
// D fp32, A/B bf16, M = 128, N = n; b_mn = 1 when B is MN-major.
__device__ __forceinline__ uint32_t umma_idesc(int n, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(b_mn) << 16) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(128 >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void named_sync(int id, int threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// (a * s + c) and a + b for two packed fp32 values: one issue slot instead of two, the same two roundings
__device__ __forceinline__ void fma2(float& lo, float& hi, uint32_t a0, uint32_t a1, float s, float c) {
  asm("{\n\t.reg .b64 a, s, c, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 s, {%4, %4};\n\tmov.b64 c, {%5, %5};\n\t"
      "fma.rn.f32x2 d, a, s, c;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "=f"(lo), "=f"(hi) : "r"(a0), "r"(a1), "f"(s), "f"(c));
}
__device__ __forceinline__ void add2(float& lo, float& hi, float b0, float b1) {
  asm("{\n\t.reg .b64 a, b, d;\n\t"
      "mov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\t"
      "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "+f"(lo), "+f"(hi) : "f"(b0), "f"(b1));
}
// True in one lane of the (converged) warp, always the same one.  Unlike a lane-id comparison it tells the compiler that the
// guarded code runs in a single lane, so MMA and TMA operands stay in uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(pred));
  return pred != 0;
}

// WL: the work-list form (helper blocks; a block takes a list of tile pieces).  It is a separate instantiation so that
// the classic launch carries none of its state through the step loop.
// VH: the value ring holds units of 64 tokens (half a step) - instantiated only where shared memory has room for
// one whole value stage but not for two.
// SP: the split-context form (clusters of NS blocks, see below).  The merge has an instantiation of its own: compiled into the
// classic form, which never takes it, it costs the step loop 6 .. 12 % through ptxas' schedule alone.
template <int HD, int RK, int RV, bool WL = false, bool VH = false, bool SP = false>
__global__ void __launch_bounds__(PTC_THREADS, 1)
lr_attend_prefill_tc_kernel(const __grid_constant__ PrefillTcMaps maps, const __grid_constant__ PrefillTcParams p) {
  using C = PrefillTcCfg<HD, RK, RV>;
  // The MMA sums the denominator.  Not in the work-list form, which would spill.  In the split-context form at head_dim 128 it slows the
  // step loop that ptxas makes of the other ranks: geometric mean of 36 turns of 32 .. 700 tokens over 8000 .. 65000 per layout, against
  // the pulling form, summed by the MMA / by the threads: ranks 32 / 32 contiguous 0.924 / 1.017, paged 0.954 / 0.945; 16 / 16 1.012 / 0.934 and
  // 0.980 / 0.934; 8 / 8 1.006 / 0.936 and 0.979 / 0.938; 0 / 16 0.968 / 0.925 and 0.972 / 0.935; 0 / 32 0.950 / 0.935 and 0.973 / 0.945.
  constexpr bool L_MMA = C::L_ROUNDED && !WL && !(SP && HD == 128 && RK != 32);
  // Running maxima over a row's 128 scores of a step (their number changes no bit).  A chain of 16 or 32 maxima keeps fewer registers than four
  // of them beside the scores, eight keep the chain short; which one ptxas makes the faster step loop of differs by form.  Whole
  // contexts, 80 turns of 360 .. 1400 tokens over 0 .. 40000 per pair of ranks, geometric mean and slowest against the kernel before the
  // MMA summed the denominator, at 2 / 4 / 8: head_dim 128 ranks 0 / 32 paged 0.962, 1.03 / 1.002, 1.08 / 0.989, 1.07; 16 / 16 contiguous
  // 0.983, 1.09 / 0.982, 1.08 / 0.958, 1.02; 32 / 32 0.952, 1.04 / 0.947, 1.05 / 0.943, 1.01; head_dim 64 ranks 0 / 64 1.003, 1.05 / 1.031,
  // 1.17 / 1.000, 1.05; 32 / 32 0.946 / 0.932 / 0.945.
  constexpr int N_MAX = SP || WL ? 4 : HD == 128 ? (RK > 0 ? 8 : 2) : RV == 64 ? 2 : 4;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);   // (pointer arithmetic, so that it stays a shared-memory address)
  const uint32_t q_u32 = smem_u32(smem);
  const uint32_t qx_u32 = q_u32 + C::Q_BYTES;
  const uint32_t kring_u32 = qx_u32 + C::QX_BYTES;
  const int KS = p.k_stages, VS = p.v_stages;
  unsigned char* vring = smem + C::Q_BYTES + C::QX_BYTES + (size_t)KS * C::KSTAGE;
  const uint32_t vring_u32 = kring_u32 + KS * C::KSTAGE;
  constexpr int vunit = VH ? C::VSTAGE / 2 : C::VSTAGE;   // bytes of one slot of the value ring
  uint64_t* bars = reinterpret_cast<uint64_t*>(vring + (size_t)VS * vunit);
  const uint32_t bar0 = smem_u32(bars);
  const uint32_t k_full = bar0, k_empty = k_full + 8 * KS, v_full = k_empty + 8 * KS, v_empty = v_full + 8 * VS,
                 s_full = v_empty + 8 * VS, s_free = s_full + 16, p_full = s_free + 16, pv_done = p_full + 16, q_full = pv_done + 16,
                 fold_done = q_full + 8, q_ready = fold_done + 8, u_full = q_ready + 8, uv_done = u_full + 8;
  const int n_bars = 2 * KS + 2 * VS + PTC_FIXED_BARS;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + n_bars);
  const uint32_t merge_bar = bar0 + 8 * (n_bars + 1);            // SP: bytes of the peers' partials
  float* xch = reinterpret_cast<float*>(bars + n_bars + 2);      // [2][128] reference maxima (by step parity) | [2][128] partial denominators

  // sixteen rows of sixteen ones, the B operand of the denominator, in the place of the partial denominators
  uint32_t* ones = reinterpret_cast<uint32_t*>(xch + 256) + ((0u - smem_u32(xch + 256)) & 255u) / 4;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = p.group;
  // Short turns over long contexts: the 128-token steps of a (row tile, kv head) are split over the NS
  // blocks of a cluster (grid/cluster z; any size from 2 to 8), each producing a partial (m, l, O) that the cluster merges
  // over distributed shared memory.
  uint32_t split, NS;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(split));
  asm volatile("mov.u32 %0, %%cluster_nctaid.z;\n" : "=r"(NS));
  // work-list tables behind the exchange area: tail[x] | pre[x] | scalars | pieces {tile, first step, steps, -}
  int* tab_tail = reinterpret_cast<int*>(xch + 4 * 128);
  int* tab_pre = tab_tail + PTC_MAX_XT;
  int* tab_sc = tab_pre + PTC_MAX_XT;                      // [0] pieces of this block, [1] sum of the tails of one kv head, [2] tail steps per helper, [3] ticket
  int* tab_seg = tab_sc + 8;
  auto steps_of = [&](int x) { return (p.T + min(p.S, (x + 1) * p.tok_per_tile) + PTC_TOK - 1) / PTC_TOK; };

  auto init_bars = [&]() {
    for (int s = 0; s < KS; ++s) { mbar_init(k_full + 8 * s, 1); mbar_init(k_empty + 8 * s, 1); }
    for (int s = 0; s < VS; ++s) { mbar_init(v_full + 8 * s, 1); mbar_init(v_empty + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(s_full + 8 * b, 1);
      mbar_init(s_free + 8 * b, PTC_SOFTMAX_WARPS / 2);
      mbar_init(p_full + 8 * b, PTC_SOFTMAX_WARPS / 2);
      mbar_init(pv_done + 8 * b, 1);                       // by step parity: a warpgroup may wait for step j-1 while step j-2 is still running
    }
    mbar_init(q_full, 1);
    mbar_init(fold_done, 1);
    mbar_init(q_ready, PTC_SOFTMAX_WARPS);
    mbar_init(u_full, PTC_SOFTMAX_WARPS);
    mbar_init(uv_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fence_async_smem();
  };
  // rows of the tile that each block finishes when the context is split over a cluster
  auto merge_share = [&](int live_rows) { return (live_rows + (int)NS - 1) / (int)NS; };
  if (threadIdx.x == 0) {
    if constexpr (SP) {
      mbar_init(merge_bar, 1);
      const int t0 = (p.longest_first ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x) * p.tok_per_tile;
      const int live = min(p.tok_per_tile, p.S - t0) * G, R = merge_share(live);
      mbar_expect_tx(merge_bar, (uint32_t)(((int)NS - 1) * max(0, min(R, live - (int)split * R)) * C::SPLIT_XS * 4));   // the one arrival, and the bytes to come
    }
    init_bars();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_holder)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if constexpr (L_MMA) {
    if (threadIdx.x < 128) { ones[threadIdx.x] = 0x3f803f80u; fence_async_smem(); }
  }
  if constexpr (WL) {
    for (int x = threadIdx.x; x < p.row_tiles; x += blockDim.x) tab_tail[x] = max(0, steps_of(x) - p.helper_p);
  }
  if (threadIdx.x < 7) {                                   // the tensor maps' first fetch would otherwise delay the first copies
    const CUtensorMap* m = &maps.k + threadIdx.x;
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(m) : "memory");
  }
  // All of the above overlaps the end of the kernel before this one (programmatic dependent launch): its whole last part
  // behind decode, combine and few-row projections, which let a dependent launch start early, launch travel and drain behind
  // the others.  Nothing of the caches, the queries or the block table is touched before that kernel has finished.  No early
  // launch of the kernel behind it: the clusters of a projection placed on the SMs that this grid leaves idle keep the rest
  // of them from fitting into one wave (301 new tokens, 80 blocks: 61.6 against 59.1 us a turn).
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  const int n_base_tiles = p.row_tiles * p.n_kv;           // work-list launch: blocks below this index own a tile
  if constexpr (WL) {
    if (threadIdx.x == 0) {
      const int X = p.row_tiles;
      int acc = 0;
      for (int x = 0; x < X; ++x) { tab_pre[x] = acc; acc += tab_tail[x]; }
      const int tail_sum = acc, total = acc * p.n_kv;
      const int per = max(1, (total + p.n_helpers - 1) / max(1, p.n_helpers));
      int n = 0;
      const int b = blockIdx.x;
      if (b < n_base_tiles) {
        const int x = b % X;
        tab_seg[0] = b; tab_seg[1] = 0; tab_seg[2] = steps_of(x) - tab_tail[x];
        n = 1;
      } else {
        const int h = b - n_base_tiles;
        int pos = min(total, h * per);
        const int hi = min(total, pos + per);
        if (pos < hi) {
          int gg = pos / tail_sum, off = pos - gg * tail_sum, x = 0;
          while (tab_pre[x] + tab_tail[x] <= off) ++x;
          while (pos < hi && n < PTC_MAX_SEG) {
            const int take = min(hi - pos, tab_pre[x] + tab_tail[x] - off);
            tab_seg[4 * n] = gg * X + x;
            tab_seg[4 * n + 1] = steps_of(x) - tab_tail[x] + (off - tab_pre[x]);
            tab_seg[4 * n + 2] = take;
            ++n; pos += take; off += take;
            while (x < X && tab_pre[x] + tab_tail[x] <= off) ++x;
            if (x == X) { ++gg; off = 0; x = 0; while (x < X - 1 && tab_tail[x] == 0) ++x; off = tab_pre[x]; }
          }
        }
      }
      tab_sc[0] = n; tab_sc[1] = tail_sum; tab_sc[2] = per;
    }
    __syncthreads();
  }
  // What this block works on.  Classic launch: one (row tile, kv head) per block, fixed for the whole kernel; `jb` is its
  // first step, `n_tiles` its number of steps (possibly zero under a context split).  Work-list launch: a short list of
  // tile pieces, taken one after the other with the block drained in between.  Loop indices are local, token
  // positions use jb + j.
  auto nseg = [&]() -> int { return WL ? tab_sc[0] : 1; };
  int g = 0, tok0 = 0, n_tok = 0, t_end = 0, full_vis = 0, jb = 0, n_tiles = 0;
  bool to_ws = false;                                      // work-list launch: this piece goes to a record
  int tile_u = 0, rec_id = 0, n_src = 1, src_first = 0;    // its tile, its record, and which records make up the tile
  auto load_piece = [&](int seg) {
    if constexpr (WL) {
      tile_u = tab_seg[4 * seg]; jb = tab_seg[4 * seg + 1]; n_tiles = tab_seg[4 * seg + 2];
      const int x = tile_u % p.row_tiles;
      g = tile_u / p.row_tiles;
      tok0 = x * p.tok_per_tile;
      to_ws = false; n_src = 1;
      if (tab_tail[x] > 0) {
        const int a_u = g * tab_sc[1] + tab_pre[x], per = tab_sc[2];
        const int hf = a_u / per, hl = (a_u + tab_tail[x] - 1) / per;
        to_ws = true;
        n_src = 2 + hl - hf;
        src_first = n_base_tiles + tile_u + hf;            // record of the first helper piece; the tile's own block writes record tile_u
        rec_id = (int)blockIdx.x < n_base_tiles ? tile_u : n_base_tiles + tile_u + ((int)blockIdx.x - n_base_tiles);
      }
    } else {
      g = blockIdx.y;
      tok0 = (p.longest_first ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x) * p.tok_per_tile;
    }
    n_tok = min(p.tok_per_tile, p.S - tok0);               // new tokens handled by this block
    t_end = p.T + tok0 + n_tok;                            // context + causal reach of the last row
    full_vis = p.T + tok0 + 1;                             // tokens visible to every row of the block
    if constexpr (!WL) {
      const int n_total = (t_end + PTC_TOK - 1) / PTC_TOK;
      const int chunk_steps = (n_total + (int)NS - 1) / (int)NS;
      jb = min(n_total, (int)split * chunk_steps);
      n_tiles = min(n_total, jb + chunk_steps) - jb;
    }
  };
  // End of a work-list piece: once every warp is here nothing of it is in flight any more (every load consumed, every
  // MMA retired); the next piece gets fresh barriers.
  auto end_piece = [&](int seg) {
    if constexpr (WL) {
      tc_fence_before();
      __syncwarp();
      named_sync(0, PTC_THREADS);
      if (seg + 1 < nseg() && threadIdx.x == 0) {
        for (int i = 0; i < n_bars; ++i) asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(bar0 + 8 * i) : "memory");
        init_bars();
      }
      __syncwarp();
      named_sync(0, PTC_THREADS);
      tc_fence_after();
    }
  };

  if (warp < PTC_FIRST_SM_WARP || warp >= PTC_FIRST_HELPER) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(PTC_CTL_REGS));
    for (int seg = 0; seg < nseg(); ++seg) {
      load_piece(seg);
      const int n_pages = (t_end + PAGE - 1) / PAGE;       // logical pages this tile may touch
      // physical block of a logical page (paged caches), fetched a step ahead of its use: the producers would otherwise sit
      // through one global round trip per step
      auto lookup = [&](int lt) -> int { return lt < n_pages ? __ldg(p.block_table + lt) : 0; };
      auto checked = [&](int ph) -> int {
        if (ph >= 0 && ph < p.n_blocks) return ph;
        atomicOr(p.status, StatusBits::BAD_INDEX);
        return 0;
      };
      // helper warps copy the pages' second slab (12: keys, 13: values) and LR rows (14, 15).  One that has nothing to copy
      // (whole-stage boxes, head_dim 64, no adapter on its side) must not walk the ring: a stage is full without it, so
      // nothing keeps the ring from going round twice before it looks, and then its wait by parity never ends.
      const int role = warp < PTC_FIRST_SM_WARP ? warp : (warp & 1) ? 3 : 0;
      const int share = warp < PTC_FIRST_SM_WARP ? 0 : 1 + ((warp - PTC_FIRST_HELPER) >> 1);
      auto copies = [&](bool whole, int rank) { return share == 0 || (!whole && (share == 1 ? C::SLABS > 1 : rank > 0)); };
      if (role == 0) {
        // -------------------------------------------------------------- TMA producer: query tile, B slices, keys
        const bool whole = p.contig || p.k_logical;
        if (share == 0) {
        const int q_rows = p.tok_per_tile * G;
        for (int i = q_rows * (HD / 8) + lane; i < 128 * (HD / 8); i += 32)    // rows no query maps to (128 not a multiple of G)
          *reinterpret_cast<uint4*>(smem + ((i % (HD / 8)) / 8) * C::SLAB_BYTES + (i / (HD / 8)) * 128 + (i % 8) * 16) = make_uint4(0, 0, 0, 0);
        fence_async_smem();
        __syncwarp();
        if (elect_one()) {
          mbar_expect_tx(q_full, q_rows * HD * 2 + (RK > 0 ? C::RKP * HD * 2 : 0));
#pragma unroll
          for (int sl = 0; sl < C::SLABS; ++sl) tma_load_3d(q_u32 + sl * C::SLAB_BYTES, &maps.q, sl * 64, g * G, tok0, q_full);
          if constexpr (RK > 0) {
            // the last key stage is the staging area of B_k until the query fold is done
#pragma unroll
            for (int sl = 0; sl < C::SLABS; ++sl)
              tma_load_2d(kring_u32 + (KS - 1) * C::KSTAGE + sl * (C::RKP * 128), &maps.bk, g * HD + sl * 64, 0, q_full);
          }
        }
        __syncwarp();
        }
        int ph_next = whole || lane >= PTC_TOK / PAGE ? 0 : lookup(jb * (PTC_TOK / PAGE) + lane);
        const int n_items = copies(whole, RK) ? n_tiles + (share == 0 && RV > 0 && n_tiles > 0 ? 1 : 0) : 0;
        for (int j = 0; j < n_items; ++j) {
          const int s = j % KS;
          if (j >= KS) mbar_wait(k_empty + 8 * s, ((j / KS) - 1) & 1, p.status);
          if (RK > 0 && j == KS - 1) mbar_wait(fold_done, 0, p.status);
          const uint32_t st = kring_u32 + (uint32_t)s * C::KSTAGE;
          const uint32_t full = k_full + 8 * s;
          __syncwarp();
          if constexpr (RV > 0) {
            if (j == n_tiles) {                            // behind the last step: the B_v slice of the value-side fold
              if (elect_one()) {
                mbar_expect_tx(full, C::BV_BYTES);
#pragma unroll
                for (int sl = 0; sl < C::SLABS; ++sl) tma_load_2d(st + sl * (C::RVP * 128), &maps.bv, g * HD + sl * 64, 0, full);
              }
              __syncwarp();
              break;
            }
          }
          if (lane == 0 && share == 0) PTC_STAMP(p, j, 8); // stage of step j free: loads go out now
          if (whole) {
            // consecutive physical blocks: one box per 64-column slab covers all eight pages of the stage
            // (4-D map [block][kv head][16][hd]); blocks past the cache end arrive as zeros
            if (elect_one()) {
              mbar_expect_tx(full, (PTC_TOK / PAGE) * C::K_PAGE_TX);
              const int blk0 = (p.k_logical ? 0 : p.first_block) + (jb + j) * (PTC_TOK / PAGE);
#pragma unroll
              for (int sl = 0; sl < C::SLABS; ++sl) tma_load_4d(st + sl * C::SLAB_BYTES, &maps.k, sl * 64, 0, g, blk0, full);
              if constexpr (RK > 0) tma_load_2d(st + C::KV_BYTES, &maps.lk, 0, blk0 * PAGE, full);
            }
            __syncwarp();
            continue;
          }
          const int live = min(PTC_TOK / PAGE, n_pages - (jb + j) * (PTC_TOK / PAGE));
          if (share == 0 && lane == 0) mbar_expect_tx(full, live * C::K_PAGE_TX);   // for all three issuers of the stage
          __syncwarp();
          if (lane < live) {
            const int ph = checked(ph_next);
            const int row_kv = (ph * p.n_kv + g) * PAGE;
#pragma unroll
            for (int sl = 0; sl < C::SLABS; ++sl)
              if (share == sl) tma_load_2d(st + sl * C::SLAB_BYTES + lane * PAGE * 128, &maps.k, sl * 64, row_kv, full);
            if constexpr (RK > 0)
              if (share == 2) tma_load_2d(st + C::KV_BYTES + lane * PAGE * C::RKP * 2, &maps.lk, 0, ph * PAGE, full);
          }
          if (lane < PTC_TOK / PAGE) ph_next = lookup((jb + j + 1) * (PTC_TOK / PAGE) + lane);
          __syncwarp();
        }
      } else if (role == 3) {
        // -------------------------------------------------------------- TMA producer: values, in units of a step or half a step
        constexpr int UT = VH ? PTC_TOK / 2 : PTC_TOK, UPG = UT / PAGE, UPS = PTC_TOK / UT, USLAB = UT * 128;
        int ph_next = p.contig || lane >= UPG ? 0 : lookup(UPS * jb * UPG + lane);
        const int n_units = copies(p.contig, RV) ? UPS * n_tiles : 0;
        for (int u = 0; u < n_units; ++u) {
          const int s = u % VS;
          if (u >= VS) mbar_wait(v_empty + 8 * s, ((u / VS) - 1) & 1, p.status);
          __syncwarp();
          if (lane == 0 && share == 0) PTC_STAMP(p, u, 9);
          const int pg0 = (UPS * jb + u) * UPG;            // first logical page of the unit
          const uint32_t st = vring_u32 + (uint32_t)s * vunit;
          const uint32_t full = v_full + 8 * s;
          if (p.contig) {
            if (elect_one()) {
              mbar_expect_tx(full, UPG * C::V_PAGE_TX);
              const int blk0 = p.first_block + pg0;
#pragma unroll
              for (int sl = 0; sl < C::SLABS; ++sl) tma_load_4d(st + sl * USLAB, &maps.v, sl * 64, 0, g, blk0, full);
              if constexpr (RV > 0) tma_load_2d(st + C::SLABS * USLAB, &maps.lv, 0, blk0 * PAGE, full);
            }
            __syncwarp();
            continue;
          }
          const int live = max(0, min(UPG, n_pages - pg0));
          if (share == 0 && lane == 0) mbar_expect_tx(full, live * C::V_PAGE_TX);       // no live page: the phase completes at once
          __syncwarp();
          if (lane < live) {
            const int ph = checked(ph_next);
            const int row_kv = (ph * p.n_kv + g) * PAGE;
#pragma unroll
            for (int sl = 0; sl < C::SLABS; ++sl)
              if (share == sl) tma_load_2d(st + sl * USLAB + lane * PAGE * 128, &maps.v, sl * 64, row_kv, full);
            if constexpr (RV > 0)
              if (share == 2) tma_load_2d(st + C::SLABS * USLAB + lane * PAGE * 128, &maps.lv, 0, ph * PAGE, full);
          }
          if (lane < UPG) ph_next = lookup(pg0 + UPG + lane);
          __syncwarp();
        }
      } else if (role == 1) {
        // -------------------------------------------------------------- S = Q' K'^T issuer
        // One thread issues these MMAs and another (warp 2) the P V' ones: an MMA costs its issuing thread
        // on the order of a hundred cycles, so two issue streams are needed to keep the tensor pipe fed.
        // All descriptors are prepared once (the address field holds addr >> 4, so moving to another
        // stage, slab or k-step is one 64-bit add of a small constant).
        const uint32_t id_s = umma_idesc(PTC_TOK, 0);
        const uint64_t qd0 = umma_desc_kmajor(q_u32, 128);
        const uint64_t qxd0 = RK > 0 ? umma_desc_kmajor(qx_u32, C::RKP * 2) : 0;
        const uint64_t kd0 = umma_desc_kmajor(kring_u32, 128);
        const uint64_t lkd0 = RK > 0 ? umma_desc_kmajor(kring_u32 + C::KV_BYTES, C::RKP * 2) : 0;
        mbar_wait(q_full, 0, p.status);
        tc_fence_after();
        __syncwarp();
        if constexpr (RK > 0) {
          // the key-side fold Q B_k^T (128 x RKP x HD): the product lands in the first columns of S buffer 0, from
          // where the softmax threads scale it into the folded-query tile
          if (elect_one()) {
            const uint32_t id_f = umma_idesc(C::RKP, 0);
            const uint64_t bd0 = umma_desc_kmajor(kring_u32 + (uint32_t)(KS - 1) * C::KSTAGE, 128);
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
              const uint64_t qo = (uint64_t)(((ks / 4) * C::SLAB_BYTES + (ks % 4) * 32) >> 4);
              const uint64_t bo = (uint64_t)(((ks / 4) * (C::RKP * 128) + (ks % 4) * 32) >> 4);
              umma_bf16(tmem_base, qd0 + qo, bd0 + bo, id_f, ks ? 1u : 0u);
            }
            umma_commit(fold_done);
          }
          __syncwarp();
          mbar_wait(q_ready, 0, p.status);
        }
        for (int j = 0; j < n_tiles; ++j) {
          const int s = j % KS;
          // S buffer j&1 is free once its warpgroup has pulled the scores of step j-2 into registers
          // (P has its own columns), so Q K^T runs up to two steps ahead of the softmax
          if (j >= 2) mbar_wait(s_free + 8 * (j & 1), ((j >> 1) - 1) & 1, p.status);
          mbar_wait(k_full + 8 * s, (j / KS) & 1, p.status);
          tc_fence_after();
          __syncwarp();
          if (lane == 0) PTC_STAMP(p, j, 10);              // keys of step j have landed (seen by the issuer)
          if (elect_one()) {
            const uint64_t so = (uint64_t)((s * C::KSTAGE) >> 4);
            const uint32_t d = tmem_base + (j & 1) * PTC_TOK;
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
              const uint64_t off = (uint64_t)(((ks / 4) * C::SLAB_BYTES + (ks % 4) * 32) >> 4);
              umma_bf16(d, qd0 + off, kd0 + so + off, id_s, ks ? 1u : 0u);
            }
            if constexpr (RK > 0) {
#pragma unroll
              for (int ks = 0; ks < C::RKP / 16; ++ks) umma_bf16(d, qxd0 + (uint64_t)(ks * 2), lkd0 + so + (uint64_t)(ks * 2), id_s, 1u);
            }
            umma_commit(k_empty + 8 * s);                  // the key stage is free as soon as S is computed
            umma_commit(s_full + 8 * (j & 1));
          }
          __syncwarp();
          if (lane == 0) PTC_STAMP(p, j, 2);               // Q K^T of step j issued
        }
      } else {
        // -------------------------------------------------------------- O' += P V' issuer
        constexpr int UT = VH ? PTC_TOK / 2 : PTC_TOK, UPS = PTC_TOK / UT, USLAB = UT * 128;
        const uint32_t id_o = umma_idesc(C::OW, 1);
        const uint64_t vd0 = umma_desc_mnmajor(vring_u32, 128, USLAB);
        const uint32_t od = tmem_base + C::TMEM_O;
        const uint32_t id_l = umma_idesc(16, 0);
        const uint64_t onesd = umma_desc_kmajor(smem_u32(ones), 32);
        for (int j = 0; j < n_tiles; ++j) {
          const int n_live = min(PTC_TOK, t_end - (jb + j) * PTC_TOK);     // tokens of this step that exist
#pragma unroll
          for (int part = 0; part < UPS; ++part) {
            const int u = UPS * j + part, s = u % VS;
            const int live_u = UPS == 1 ? n_live : max(0, min(UT, n_live - part * UT));
            mbar_wait(v_full + 8 * s, (u / VS) & 1, p.status);
            if (lane == 0) PTC_STAMP(p, j, 11);            // values of step j have landed
            if (live_u < UT && (p.contig || (live_u % PAGE) != 0)) {
              // value rows past the end may hold anything (the rest of a partly written page; with whole-stage
              // boxes also the pages behind it), and 0 * NaN would poison the accumulators: clear them
              // before the MMA reads the stage
              unsigned char* ub = vring + (size_t)s * vunit;
              const int r1 = p.contig ? UT : (live_u + PAGE - 1) / PAGE * PAGE;
              for (int r = live_u; r < r1; ++r)
                for (int sl = 0; sl < C::VSLABS; ++sl)
                  for (int c = lane; c < 8; c += 32) *reinterpret_cast<uint4*>(ub + sl * USLAB + r * 128 + c * 16) = make_uint4(0, 0, 0, 0);
              fence_async_smem();
              __syncwarp();
            }
            if (part == 0) mbar_wait(p_full + 8 * (j & 1), (j >> 1) & 1, p.status);
            tc_fence_after();
            __syncwarp();
            if (lane == 0) PTC_STAMP(p, j, 0);             // P of step j seen by the P V' issuer
            if (elect_one()) {
              const uint32_t a = tmem_base + C::TMEM_P + (C::PB == 2 ? (j & 1) * 64 : 0) + part * (UT / 2);  // packed bf16 P, 2 per column
              const uint64_t so = (uint64_t)((s * vunit) >> 4);
              if (live_u == UT) {
#pragma unroll
                for (int ks = 0; ks < UT / 16; ++ks) {
                  umma_bf16_ts(od, a + ks * 8, vd0 + so + (uint64_t)(ks * 128), id_o, (j | part | ks) ? 1u : 0u);
                  if constexpr (L_MMA) umma_bf16_ts(od + C::OW, a + ks * 8, onesd, id_l, (j | part | ks) ? 1u : 0u);
                }
              } else {
                const int n_ks = (live_u + 15) / 16;
                for (int ks = 0; ks < n_ks; ++ks) {
                  umma_bf16_ts(od, a + ks * 8, vd0 + so + (uint64_t)(ks * 128), id_o, (j | part | ks) ? 1u : 0u);
                  if constexpr (L_MMA) umma_bf16_ts(od + C::OW, a + ks * 8, onesd, id_l, (j | part | ks) ? 1u : 0u);
                }
              }
              umma_commit(v_empty + 8 * s);
              if (part == UPS - 1) umma_commit(pv_done + 8 * (j & 1));
            }
            __syncwarp();
            if (lane == 0) PTC_STAMP(p, j, 1);             // P V' of step j issued
          }
        }
        if constexpr (RV > 0) {
          if (n_tiles > 0) {
            // the value-side fold O += (s_v U) B_v: three bf16 terms of s_v U in TMEM columns 0.., B_v as one more "value stage"
            const int s = n_tiles % KS;
            mbar_wait(k_full + 8 * s, (n_tiles / KS) & 1, p.status);
            mbar_wait(u_full, 0, p.status);
            tc_fence_after();
            __syncwarp();
            if (elect_one()) {
              const uint32_t id_u = umma_idesc(HD, 1);
              const uint64_t bvd = umma_desc_mnmajor(kring_u32 + (uint32_t)s * C::KSTAGE, 128, C::RVP * 128);
#pragma unroll
              for (int t = 0; t < 3; ++t)
#pragma unroll
                for (int ks = 0; ks < C::RVP / 16; ++ks)
                  umma_bf16_ts(od, tmem_base + t * C::UPW + ks * 8, bvd + (uint64_t)(ks * 128), id_u, 1u);
              umma_commit(uv_done);
            }
            __syncwarp();
          }
        }
      }
      __syncwarp();
      if constexpr (SP) { cluster_barrier(); cluster_barrier(); }     // the softmax warps' merge of the context splits
      end_piece(seg);
    }
  } else {
    // ------------------------------------------------------------------ softmax / correction / epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(PTC_SM_REGS));
    constexpr int NSM = PTC_SOFTMAX_WARPS * 32;                   // softmax threads
    const int quad = warp & 3;                                    // TMEM lane quadrant this warp may touch
    const int wg = (warp - PTC_FIRST_SM_WARP) >> 2;               // warpgroup: steps of this parity; in the epilogue, every other chunk of columns
    const int row = quad * 32 + lane;                             // query row of this thread
    const int tid = (warp - PTC_FIRST_SM_WARP) * 32 + lane;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
    float* mref = xch;                                            // [2][128]: reference maximum after a step, by step parity
    float* lpart = xch + 256;                                     // [2][128]: the warpgroups' denominators
    const int bar_in = 2 + 2 * quad + (wg ^ 1), bar_out = 2 + 2 * quad + wg;   // named barriers: hand-over of the reference maximum within a warp pair
    for (int seg = 0; seg < nseg(); ++seg) {
      load_piece(seg);
      PTC_WL_STAMP(p, seg, 0);                                     // piece starts
      // tokens visible to this thread's row, and to every row of the block, counted from the piece's first step
      const int lim = (row < n_tok * G ? p.T + tok0 + row / G + 1 : 0) - jb * PTC_TOK, full = full_vis - jb * PTC_TOK;
      if constexpr (RK > 0) {
        // the folded query: fp32 product of the fold MMA, scaled and rounded to bf16, as a K-major swizzled operand
        constexpr int CPR = C::RKP / 8;
        mbar_wait(fold_done, 0, p.status);
        tc_fence_after();
#pragma unroll 1
        for (int c = wg; c < C::RKP / 16; c += 2) {                // 16 coordinates per pass
          uint32_t fv[16];
          tmem_ld16(lane_addr + c * 16, fv);
          tmem_wait_ld();
          uint32_t pk[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) pk[k] = pack_bf16(__uint_as_float(fv[2 * k]) * p.s_k, __uint_as_float(fv[2 * k + 1]) * p.s_k);
          *reinterpret_cast<uint4*>(smem + C::Q_BYTES + swz_off<CPR>(row, 2 * c)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          *reinterpret_cast<uint4*>(smem + C::Q_BYTES + swz_off<CPR>(row, 2 * c + 1)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        }
        tc_fence_before();                                        // the reads of S buffer 0 precede the first Q K^T
        fence_async_smem();                                       // generic-proxy writes -> visible to the MMA unit
        __syncwarp();
        if (lane == 0) mbar_arrive(q_ready);
      } else {
        mbar_wait(q_full, 0, p.status);                           // (a block without steps must not reuse the query tile before it has landed)
      }
      PTC_WL_STAMP(p, seg, 1);                                     // query tile loaded and folded

      float m_own = NEG_BIG, l_sum = 0.f;                         // reference and denominator of this warpgroup's steps
      // One step of the online softmax: this thread's row, all 128 scores.  MASKED is a compile-time flag so
      // that the common step (far from the causal edge) carries no per-element compare/select.
      auto step = [&](int j, auto masked_tag) {
        constexpr bool MASKED = decltype(masked_tag)::value;
        uint32_t sv[4][32];
        mbar_wait(s_full + 8 * wg, (j >> 1) & 1, p.status);
        tc_fence_after();
        if ((tid & 127) == 0) PTC_STAMP(p, j, 4);                  // scores of step j seen
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(lane_addr + wg * PTC_TOK + c * 32, sv[c]);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(s_free + 8 * wg);               // the S buffer may be overwritten
        if ((tid & 127) == 0) PTC_STAMP(p, j, 7);                  // scores in registers
        if constexpr (MASKED) {
          const int nvis = lim - j * PTC_TOK;           // visible tokens of this step
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int k = 0; k < 32; ++k)
              if (c * 32 + k >= nvis) sv[c][k] = 0xff800000u;      // -inf: weight zero
        }
        float tm[N_MAX];
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) tm[i] = -INFINITY;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int k = 0; k < 32; k += 2)                          // two elements per step: the three-input maximum
            tm[(k >> 1) & (N_MAX - 1)] = fmaxf(tm[(k >> 1) & (N_MAX - 1)], fmaxf(__uint_as_float(sv[c][k]), __uint_as_float(sv[c][k + 1])));
#pragma unroll
        for (int n = N_MAX / 2; n > 0; n /= 2)
#pragma unroll
          for (int i = 0; i < n; ++i) tm[i] = fmaxf(tm[i], tm[i + n]);
        const float tmax = tm[0] * p.scale_log2;
        float m_prev = NEG_BIG;                                    // the reference in force before this step
        if (j > 0) {
          named_sync(bar_in, 64);
          m_prev = mref[(wg ^ 1) * 128 + row];
        }
        const float m_new = tmax > m_prev + PTC_RAISE ? tmax : m_prev;
        mref[wg * 128 + row] = m_new;
        if (j + 1 < n_tiles) named_arrive(bar_out, 64);
        if ((tid & 127) == 0) PTC_STAMP(p, j, 5);                  // reference maximum settled
        if (j > 0 && __any_sync(0xffffffffu, m_new != m_prev)) {
          const float alpha = fast_exp2(m_prev - m_new);           // 1 for rows that keep their maximum
          // O' is complete through step j-1.  A wait names a phase by its parity, so it holds only on a barrier that is in that
          // phase or the next one: step j-3, the one before on this barrier, has to have retired first.  That follows from
          // step j-2, whose own barrier cannot be further (step j is not published); waiting for step j-3 itself
          // would never end where step j-1 has retired already.  (With one P buffer this warpgroup's previous step
          // waited for exactly that.)
          if (C::PB == 2 && j > 2) mbar_wait(pv_done + 8 * wg, ((j - 2) >> 1) & 1, p.status);
          mbar_wait(pv_done + 8 * (wg ^ 1), ((j - 1) >> 1) & 1, p.status);
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < (L_MMA ? C::OWL : C::OW) / 16; ++c) {
            uint32_t ov[16];
            tmem_ld16(lane_addr + C::TMEM_O + c * 16, ov);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) ov[k] = __float_as_uint(__uint_as_float(ov[k]) * alpha);
            tmem_st16(lane_addr + C::TMEM_O + c * 16, ov);
          }
          tmem_wait_st();
        }
        if constexpr (!L_MMA) { l_sum *= fast_exp2(m_own - m_new); m_own = m_new; }
        float ls[4] = {0.f, 0.f, 0.f, 0.f};
        const float neg_m = -m_new;
        uint32_t pk[2][32];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int k = 0; k < 32; k += 2) {
            float p0, p1;
            fma2(p0, p1, sv[c][k], sv[c][k + 1], p.scale_log2, neg_m);
            p0 = fast_exp2(p0); p1 = fast_exp2(p1);
            const uint32_t w = pack_bf16(p0, p1);
            if constexpr (L_MMA) { }                                  // (summed by the P V' issuer's second MMA)
            else if constexpr (C::L_ROUNDED) add2(ls[k & 2], ls[(k & 2) + 1], __uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
            else if constexpr (WL) { ls[k & 2] += p0; ls[(k & 2) + 1] += p1; }      // (packed, ptxas spills here)
            else add2(ls[k & 2], ls[(k & 2) + 1], p0, p1);
            pk[c >> 1][(c & 1) * 16 + k / 2] = w;
          }
        if constexpr (!L_MMA) l_sum += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        if ((tid & 127) == 0) PTC_STAMP(p, j, 14);                 // all exponentials done
        // the P buffer may be overwritten once the P V' that read it last has retired
        if (j >= C::PB) {
          const int jp = j - C::PB;
          mbar_wait(pv_done + 8 * (jp & 1), (jp >> 1) & 1, p.status);
          tc_fence_after();
        }
        if ((tid & 127) == 0) PTC_STAMP(p, j, 15);                 // that P V' has retired
        const uint32_t pcol = lane_addr + C::TMEM_P + (C::PB == 2 ? wg * 64 : 0);
        tmem_st32(pcol, pk[0]);
        tmem_st32(pcol + 32, pk[1]);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + 8 * wg);
        if ((tid & 127) == 0) PTC_STAMP(p, j, 6);                  // P published
      };
      for (int j = wg; j < n_tiles; j += 2) {
        if (j * PTC_TOK + PTC_TOK > full) step(j, std::true_type{});   // only the last few steps reach the causal edge
        else step(j, std::false_type{});
      }
      PTC_WL_STAMP(p, seg, 2);                                     // this warpgroup's steps done
      // ---- O' complete: reference maximum and denominator of the row, then the value-side fold
      float m_fin = NEG_BIG;
      named_sync(1, NSM);                                          // (also: every P is published, so at most the last two P V' are still running)
      if (n_tiles > 0) {
        m_fin = mref[((n_tiles - 1) & 1) * 128 + row];
        mbar_wait(pv_done + 8 * ((n_tiles - 1) & 1), ((n_tiles - 1) >> 1) & 1, p.status);
        tc_fence_after();
      }
      if constexpr (!L_MMA) {
        lpart[wg * 128 + row] = l_sum * fast_exp2(m_own - m_fin);
        named_sync(1, NSM);
      }
      if constexpr (WL) load_piece(seg);                           // read again rather than held in registers through the steps
      float l_tot = 0.f;
      if constexpr (L_MMA) {
        if (n_tiles > 0) {
          uint32_t lv;
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(lv) : "r"(lane_addr + C::TMEM_O + C::OW));
          tmem_wait_ld();
          l_tot = __uint_as_float(lv);
        }
      } else {
        l_tot = lpart[row] + lpart[128 + row];
      }
      if constexpr (RV > 0) {
        if (n_tiles > 0) {
          // s_v U as three bf16 terms (exact to fp32's 24 bits), packed A operand in the idle S columns
#pragma unroll 1
          for (int c = wg; c < C::RVP / 16; c += 2) {
            uint32_t uv[16], tk[3][8];
            tmem_ld16(lane_addr + C::TMEM_O + HD + c * 16, uv);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              float x0 = __uint_as_float(uv[2 * k]) * p.s_v, x1 = __uint_as_float(uv[2 * k + 1]) * p.s_v;   // (padding columns hold zeros)
#pragma unroll
              for (int t = 0; t < 3; ++t) {
                const uint32_t w = pack_bf16(x0, x1);
                tk[t][k] = w;
                x0 -= bf16_bits_to_float(w & 0xffff);
                x1 -= bf16_bits_to_float(w >> 16);
              }
            }
#pragma unroll
            for (int t = 0; t < 3; ++t) tmem_st8(lane_addr + t * C::UPW + c * 8, tk[t]);
          }
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(u_full);
          mbar_wait(uv_done, 0, p.status);
          tc_fence_after();
        }
      }
      PTC_WL_STAMP(p, seg, 3);                                     // numerator complete
      constexpr int XS = C::SPLIT_XS;
      if constexpr (SP) {
        // ---- split context: block `split` of the cluster finishes rows [split R, split R + nrows) of the tile.  A block lays its
        //      partial out by rows (O, then m and l in the padding), so that what another block finishes is one run of
        //      memory: one bulk copy per peer into that block's receive area, counted on its merge barrier.  (Pulled with 16-byte
        //      loads over distributed shared memory, 64 new tokens over 16384 spent 8.9 us from here to the end, now 5.2.)
        // Its place in the grid, and (FRESH_SMEM) where its shared memory begins, the block reads again here, through moves that the compiler
        // cannot merge with the ones above the step loop: carried through it, these registers change the schedule that
        // ptxas finds for the loop.  Against the form that pulled the partials, over 36 turns of 32 .. 700 tokens on 8000 .. 65000 per pair of ranks
        // (head_dim 128, geometric mean and slowest): ranks 16 / 16 contiguous 0.967 and 1.12 -> 0.934 and 1.00, 8 / 8 0.970 and
        // 1.15 -> 0.936 and 1.00, 0 / 32 0.945 and 1.02 -> 0.935 and 1.00, 32 / 32 0.944 and 1.03 -> 0.924 and 0.99.  The last, and rank 64,
        // do better with the shared-memory addresses carried (32 / 32: 1.017 otherwise, 0 / 64 1.00 instead of 0.975).
        constexpr bool FRESH_SMEM = HD == 64 || (RK != 32 && RV != 64);
        auto fresh = [](uint32_t x) { uint32_t y; asm volatile("mov.u32 %0, %1;\n" : "=r"(y) : "r"(x)); return y; };
        uint32_t split, NS, bx, by, tx;
        asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(split));
        asm volatile("mov.u32 %0, %%cluster_nctaid.z;\n" : "=r"(NS));
        asm volatile("mov.u32 %0, %%ctaid.x;\n" : "=r"(bx));
        asm volatile("mov.u32 %0, %%ctaid.y;\n" : "=r"(by));
        asm volatile("mov.u32 %0, %%tid.x;\n" : "=r"(tx));
        const int wm = (int)(tx >> 5) - PTC_FIRST_SM_WARP, lane = tx & 31;
        const int wg = wm >> 2, row = ((int)(tx >> 5) & 3) * 32 + lane, tid = wm * 32 + lane, g = (int)by;
        const int tok0 = (p.longest_first ? (int)(gridDim.x - 1 - bx) : (int)bx) * p.tok_per_tile, n_tok = min(p.tok_per_tile, p.S - tok0);
        unsigned char* area = smem;
        uint32_t merge_u32 = merge_bar;
        if constexpr (FRESH_SMEM) {
          const uint32_t base = fresh(smem_u32(smem_raw)), off = (0u - base) & 1023u;
          const int ks = (int)fresh(p.k_stages), vs = (int)fresh(p.v_stages);
          area = smem_raw + off;
          merge_u32 = base + off + C::Q_BYTES + C::QX_BYTES + ks * C::KSTAGE + vs * vunit + 8 * (2 * ks + 2 * vs + PTC_FIXED_BARS + 1);
        }
        const int live = n_tok * G, R = (live + (int)NS - 1) / (int)NS;
        const int nrows = max(0, min(R, live - (int)split * R));
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");   // this block's rings are idle: peers may send over them
        float* xo = reinterpret_cast<float*>(area);               // the merge area starts at the Q tile: every MMA has completed
        float* recv = xo + 128 * XS;                              // [NS - 1][R][XS], slot = sender's rank with the own rank left out
#pragma unroll 1
        for (int c = wg; c < HD / 16; c += 2) {
          uint32_t ov[16];
          if (n_tiles > 0) {
            tmem_ld16(lane_addr + C::TMEM_O + c * 16, ov);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) ov[k] = 0u;
          }
#pragma unroll
          for (int k = 0; k < 16; k += 4)
            *reinterpret_cast<uint4*>(xo + row * XS + c * 16 + k) = make_uint4(ov[k], ov[k + 1], ov[k + 2], ov[k + 3]);
        }
        if (wg == 0) *reinterpret_cast<float2*>(xo + row * XS + HD) = make_float2(m_fin, l_tot);
        fence_async_smem();                                       // the copy engine reads what these threads wrote
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
        named_sync(1, NSM);
        if (tid < (int)NS && tid != (int)split) {
          const int n = max(0, min(R, live - tid * R));
          const uint32_t dst = dsmem_addr(smem_u32(recv) + (uint32_t)(((int)split < tid ? (int)split : (int)split - 1) * R * XS * 4), tid);
          if (n > 0)
            asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                         ::"r"(dst), "r"(smem_u32(xo + tid * R * XS)), "r"(n * XS * 4), "r"(dsmem_addr(merge_u32, tid)) : "memory");
        }
        __syncwarp();
        mbar_wait_cluster(merge_u32, 0, p.status);
        __syncwarp();
        // everything addressed to this block has arrived; a peer whose copies still read its shared memory waits for this
        asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
        for (int it = tid; it < nrows * (HD / 8); it += NSM) {    // eight columns per item
          const int rl = it / (HD / 8), c8 = (it % (HD / 8)) * 8;
          const int rowg = (int)split * R + rl;
          auto src = [&](int s2) -> const float* { return s2 == (int)split ? xo + rowg * XS : recv + ((s2 < (int)split ? s2 : s2 - 1) * R + rl) * XS; };
          float wt[PTC_MAX_SPLIT], M = NEG_BIG, L = 0.f;
#pragma unroll
          for (int s2 = 0; s2 < PTC_MAX_SPLIT; ++s2) { wt[s2] = s2 < (int)NS ? src(s2)[HD] : NEG_BIG; M = fmaxf(M, wt[s2]); }
          float o[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int s2 = 0; s2 < PTC_MAX_SPLIT; ++s2) {            // split order: deterministic
            if (s2 < (int)NS) {
              const float* x = src(s2);
              const float4 a = *reinterpret_cast<const float4*>(x + c8), b = *reinterpret_cast<const float4*>(x + c8 + 4);
              const float wv = fast_exp2(wt[s2] - M);
              L += wv * x[HD + 1];
              o[0] += wv * a.x; o[1] += wv * a.y; o[2] += wv * a.z; o[3] += wv * a.w;
              o[4] += wv * b.x; o[5] += wv * b.y; o[6] += wv * b.z; o[7] += wv * b.w;
            }
          }
          const float inv = L > 0.f ? 1.f / L : 0.f;
          const int i_out = tok0 + rowg / G, h_out = rowg % G;
          uint4 w;
          w.x = pack_bf16(o[0] * inv, o[1] * inv); w.y = pack_bf16(o[2] * inv, o[3] * inv);
          w.z = pack_bf16(o[4] * inv, o[5] * inv); w.w = pack_bf16(o[6] * inv, o[7] * inv);
          *reinterpret_cast<uint4*>(p.out + ((size_t)i_out * p.n_q + (size_t)g * G + h_out) * HD + c8) = w;
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
      } else if (WL && to_ws) {
        // ---- work-list launch: this piece's partial (m, l, O) goes to its record in global memory; the block that
        //      arrives last at the tile's ticket merges the tile's records in a fixed order and writes the output
        float* rec = p.ws_rec + (size_t)rec_id * C::REC_FLOATS;
#pragma unroll 1
        for (int c = wg; c < HD / 16; c += 2) {
          uint32_t ov[16];
          tmem_ld16(lane_addr + C::TMEM_O + c * 16, ov);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 16; k += 4)
            __stcg(reinterpret_cast<uint4*>(rec + row * XS + c * 16 + k), make_uint4(ov[k], ov[k + 1], ov[k + 2], ov[k + 3]));
        }
        if (wg == 0) { __stcg(rec + 128 * XS + row, m_fin); __stcg(rec + 128 * XS + 128 + row, l_tot); }
        __threadfence();
        PTC_WL_STAMP(p, seg, 4);                                   // record written
        named_sync(1, NSM);
        if (tid == 0) tab_sc[3] = (int)atomicAdd(p.ws_ticket + tile_u, 1u);
        named_sync(1, NSM);
        if (tab_sc[3] == n_src - 1) {
          __threadfence();
          // weights over the Q tile: every load of this piece has been consumed, every MMA has retired
          float* wts = reinterpret_cast<float*>(smem);      // [n_src][128] weights of the pieces
          float* linv = wts + PTC_MAX_SRC * 128;            // [128]
          auto src = [&](int k) -> const float* {
            return p.ws_rec + (size_t)(k == 0 ? tile_u : src_first + k - 1) * C::REC_FLOATS;
          };
          if (tid < 128) {
            float ms[PTC_MAX_SRC], M = NEG_BIG, L = 0.f;
#pragma unroll
            for (int k = 0; k < PTC_MAX_SRC; ++k) { ms[k] = k < n_src ? __ldcg(src(k) + 128 * XS + tid) : NEG_BIG; M = fmaxf(M, ms[k]); }
#pragma unroll
            for (int k = 0; k < PTC_MAX_SRC; ++k) {
              if (k < n_src) {
                const float wv = fast_exp2(ms[k] - M);
                wts[k * 128 + tid] = wv;
                L += wv * __ldcg(src(k) + 128 * XS + 128 + tid);       // piece order: deterministic
              }
            }
            linv[tid] = L > 0.f ? 1.f / L : 0.f;
          }
          named_sync(1, NSM);
          constexpr int C8 = HD / 8;                        // eight columns per item
          constexpr int UN = 4;                             // items per thread in flight: the records come from L2
          for (int it0 = tid; it0 < n_tok * G * C8; it0 += NSM * UN) {
            float o[UN][8];
#pragma unroll
            for (int u = 0; u < UN; ++u)
#pragma unroll
              for (int k = 0; k < 8; ++k) o[u][k] = 0.f;
            for (int k = 0; k < n_src; ++k) {
              const float* sk = src(k);
              float4 x[UN][2];
#pragma unroll
              for (int u = 0; u < UN; ++u) {
                const int it = it0 + u * NSM;
                if (it < n_tok * G * C8) {
                  const float4* a = reinterpret_cast<const float4*>(sk + (it / C8) * XS + (it % C8) * 8);
                  x[u][0] = __ldcg(a); x[u][1] = __ldcg(a + 1);
                } else {
                  x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
              }
#pragma unroll
              for (int u = 0; u < UN; ++u) {
                const float wv = wts[k * 128 + min(127, (it0 + u * NSM) / C8)];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  o[u][4 * h] += wv * x[u][h].x; o[u][4 * h + 1] += wv * x[u][h].y;
                  o[u][4 * h + 2] += wv * x[u][h].z; o[u][4 * h + 3] += wv * x[u][h].w;
                }
              }
            }
#pragma unroll
            for (int u = 0; u < UN; ++u) {
              const int it = it0 + u * NSM;
              if (it < n_tok * G * C8) {
                const int rl = it / C8, c8 = (it % C8) * 8;
                const float inv = linv[rl];
                uint4 w;
                w.x = pack_bf16(o[u][0] * inv, o[u][1] * inv); w.y = pack_bf16(o[u][2] * inv, o[u][3] * inv);
                w.z = pack_bf16(o[u][4] * inv, o[u][5] * inv); w.w = pack_bf16(o[u][6] * inv, o[u][7] * inv);
                *reinterpret_cast<uint4*>(p.out + ((size_t)(tok0 + rl / G) * p.n_q + (size_t)g * G + rl % G) * HD + c8) = w;
              }
            }
          }
          if (tid == 0) p.ws_ticket[tile_u] = 0u;           // the workspace is ready for the next call
          PTC_WL_STAMP(p, seg, 6);                                 // merged and stored
        }
        PTC_WL_STAMP(p, seg, 5);                                   // piece ends
      } else {
        const float inv = 1.f / l_tot;
        __nv_bfloat16* orow = p.out + ((size_t)(tok0 + row / G) * p.n_q + (size_t)g * G + row % G) * HD;
#pragma unroll
        for (int c = wg; c < HD / 32; c += 2) {                   // 32-column chunks: this warpgroup's half of the row
          uint32_t ov[32];
          tmem_ld32(lane_addr + C::TMEM_O + c * 32, ov);
          tmem_wait_ld();
          if (row < n_tok * G) {
#pragma unroll
            for (int k = 0; k < 32; k += 8) {
              uint4 w;
              w.x = pack_bf16(__uint_as_float(ov[k]) * inv, __uint_as_float(ov[k + 1]) * inv);
              w.y = pack_bf16(__uint_as_float(ov[k + 2]) * inv, __uint_as_float(ov[k + 3]) * inv);
              w.z = pack_bf16(__uint_as_float(ov[k + 4]) * inv, __uint_as_float(ov[k + 5]) * inv);
              w.w = pack_bf16(__uint_as_float(ov[k + 6]) * inv, __uint_as_float(ov[k + 7]) * inv);
              *reinterpret_cast<uint4*>(orow + c * 32 + k) = w;
            }
          }
        }
      }
      end_piece(seg);
    }
  }
  tc_fence_before();
  __syncwarp();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

}  // namespace precc
