// Skinny projection GEMM on the 5th-generation tensor cores (tcgen05 + TMEM), fed by TMA.
//
//   C[M, N_out] = X[M, K] . Wt[N_out, K]^T        (both operands K-major bf16, fp32 accumulate)
//
// with a scatter epilogue that writes bf16 rows straight into the paged caches:
//   mode 0  LR precompute (Section 3.1):  column -> (projection, agent, r index), LR cache rows
//   mode 1  base projection (Section 3.2): column -> (projection, kv head, c), base cache rows
//   mode 2  both at once: the first 2*n_kv*hd columns go to the base caches, the rest to the LR caches
//           (the hidden states of a newly processed segment are read once, Section 3.1)
//
// Persistent blocks, 128 x BN output tiles.  Warp roles: warp 0 = TMA producer (one lane), warp 1 =
// TMEM owner + MMA issuer (one lane), warps 2..5 = epilogue (one TMEM lane = one row each).  A
// STAGES-deep ring of {X tile 128x64, Wt tile BNx64} in 128-byte-swizzled shared memory is handed from
// producer to issuer with mbarriers; tcgen05.commit releases a stage when its MMAs have read it.  The
// accumulator is double-buffered in TMEM (2 x BN columns), so a tile's epilogue overlaps the next
// tile's MMAs.
// Every wait is bounded: on expiry the waiter records PRECC_STATUS_TIMEOUT and carries on, so the
// kernel always terminates and frees its TMEM.
#pragma once
#include "tc_common.cuh"

namespace precc {

// Routes eight consecutive output columns [gc, gc+8) of one row (cache block `blk`, offset `off`) to
// their place in the paged caches: column -> (projection, head, c) for base columns, (projection, agent,
// r) for LR columns (skipped when the agent's bit in `mask` — the call's mask or the row's own — is clear).  Pieces never straddle a destination row
// because head_dim and the ranks are multiples of 8.
// `gm` is the row's index in the call (for the optional second LR destination of that row, see lr_copy_slots).
__device__ __forceinline__ void store_piece(const GemmParams& p, long long blk, int off, int gc, const float (&v8)[8],
                                            unsigned long long mask, int gm) {
  const int w = p.n_kv * p.hd;
  __nv_bfloat16* dst;
  __nv_bfloat16* dst2 = nullptr;
  const bool to_base = p.mode == 1 || (p.mode == 2 && gc < 2 * w);
  if (!to_base) {
    const int n_k = p.n_agents * p.rank_k;
    const int gl = p.mode == 2 ? gc - 2 * w : gc;
    const bool is_v = gl >= n_k;
    const int rr = is_v ? p.rank_v : p.rank_k;
    const int cc = is_v ? gl - n_k : gl;
    const int sh = is_v ? p.rv_shift : p.rk_shift;
    const int agent = cc >> sh, ri = cc & (rr - 1);
    if (!((mask >> agent) & 1ull)) return;
    dst = (is_v ? p.lr_v : p.lr_k) + (((long long)agent * p.n_blocks + blk) * PAGE + off) * rr + ri;
    if (p.lr_copy_slots) {
      const long long s2 = p.lr_copy_slots[gm];
      if (s2 >= p.n_blocks * PAGE) atomicOr(p.status, StatusBits::BAD_INDEX);
      else if (s2 >= 0) dst2 = (is_v ? p.lr_v : p.lr_k) + ((long long)agent * p.n_blocks * PAGE + s2) * rr + ri;
    }
  } else {
    const bool is_v = gc >= w;
    const int cc = is_v ? gc - w : gc;
    const int g = cc >> p.hd_shift, c = cc & (p.hd - 1);
    dst = (is_v ? p.base_v : p.base_k) + ((blk * p.n_kv + g) * PAGE + off) * p.hd + c;
  }
  uint4 v;
  v.x = pack_bf16(v8[0], v8[1]);
  v.y = pack_bf16(v8[2], v8[3]);
  v.z = pack_bf16(v8[4], v8[5]);
  v.w = pack_bf16(v8[6], v8[7]);
  *reinterpret_cast<uint4*>(dst) = v;
  if (dst2) *reinterpret_cast<uint4*>(dst2) = v;
}

// Epilogue of one output tile for one warp: TMEM lane = tile row (this warp owns lanes lane_base .. lane_base + 31 of
// the accumulator at `tmem_tile`, which holds rows m0 .. m0 + 127 and columns n0 .. n0 + BN - 1).  Waits for the
// accumulator (bounded), converts to bf16 and routes 16-byte pieces to the paged caches; key columns of the rotary
// variant are rotated by the row's position first.
// The epilogue shares its SM's issue slots with the lanes that feed the tensor pipe, so it is kept lean: what depends
// on the row (its slot -> element offsets into the base and LR arrays, its agent mask, its optional second LR
// destination) is computed once per tile, what depends on the column (projection, head or agent, offset inside the
// destination row) is the same for every lane and uses shifts (head_dim and the ranks are powers of two).
__device__ __forceinline__ void gemm_epilogue_tile(const GemmParams& p, uint32_t tmem_tile, int m0, int n0, int lane_base, int lane,
                                                   uint32_t acc_full_bar, uint32_t parity) {
  const int row = lane_base + lane;
  const int hs = p.hd_shift;
  const int w = p.n_kv << hs;
  const int gm = m0 + row;
  bool row_ok = gm < p.M;
  long long slot = 0;
  if (row_ok) {
    slot = p.slot_mapping ? (long long)p.slot_mapping[gm] : p.start_slot + gm;
    if (slot < 0 || slot >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); row_ok = false; slot = 0; }
  }
  const long long blk = slot / PAGE;
  const int off = (int)(slot % PAGE);
  const unsigned long long row_mask = (p.row_masks && row_ok) ? p.row_masks[gm] : p.agent_mask;
  long long slot2 = -1;                               // second destination of this row's LR pieces, if any
  if (p.lr_copy_slots && row_ok) {
    slot2 = p.lr_copy_slots[gm];
    if (slot2 >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); slot2 = -1; }
  }
  long long pos = 0;
  if (p.rope && row_ok) {
    pos = p.positions ? (long long)p.positions[gm] : p.start_pos + gm;
    if (pos < 0 || pos >= p.max_pos) { atomicOr(p.status, StatusBits::BAD_INDEX); row_ok = false; }
  }
  // element offsets of this row inside the base arrays ([blk][g][off][c]: the head term is added per column) and
  // inside one agent's LR arrays ([blk][off][r] = [slot][r])
  const long long base_row = ((blk * p.n_kv * PAGE) + off) << hs;
  const int n_k = p.n_agents << p.rk_shift;           // LR-K columns of the call (0 when rank_k == 0: n_agents << 0 is not used then)
  const int n_lrk = p.rank_k > 0 ? n_k : 0;
  mbar_wait_relaxed(acc_full_bar, parity, p.status);
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  for (int c0 = 0; c0 < p.BN && n0 + c0 < p.N_out; c0 += 16) {
    if (p.rope && n0 + c0 < w) {
      // key columns: chunk [c, c+16) of the lower half of a head together with its partner chunk
      const int gc = n0 + c0;
      const int g = gc >> hs, c = gc & (p.hd - 1);
      if (c >= p.hd / 2) continue;                  // done with its partner
      uint32_t lo[16], hi[16];
      tmem_ld16(tmem_tile + (static_cast<uint32_t>(lane_base) << 16) + c0, lo);
      tmem_ld16(tmem_tile + (static_cast<uint32_t>(lane_base) << 16) + c0 + p.hd / 2, hi);
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
      if (!row_ok) continue;
      const float4* cs = p.rope + pos * (p.hd / 4) + c / 2;
      uint32_t ol[8], oh[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 t4 = __ldg(cs + k);
        const float l0 = __uint_as_float(lo[2 * k]), l1 = __uint_as_float(lo[2 * k + 1]);
        const float h0 = __uint_as_float(hi[2 * k]), h1 = __uint_as_float(hi[2 * k + 1]);
        ol[k] = pack_bf16(l0 * t4.x - h0 * t4.y, l1 * t4.z - h1 * t4.w);
        oh[k] = pack_bf16(h0 * t4.x + l0 * t4.y, h1 * t4.z + l1 * t4.w);
      }
      __nv_bfloat16* dst = p.base_k + base_row + ((long long)(g * PAGE) << hs) + c;
      reinterpret_cast<uint4*>(dst)[0] = make_uint4(ol[0], ol[1], ol[2], ol[3]);
      reinterpret_cast<uint4*>(dst)[1] = make_uint4(ol[4], ol[5], ol[6], ol[7]);
      reinterpret_cast<uint4*>(dst + p.hd / 2)[0] = make_uint4(oh[0], oh[1], oh[2], oh[3]);
      reinterpret_cast<uint4*>(dst + p.hd / 2)[1] = make_uint4(oh[4], oh[5], oh[6], oh[7]);
      continue;
    }
    uint32_t r[16];
    tmem_ld16(tmem_tile + (static_cast<uint32_t>(lane_base) << 16) + c0, r);
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
    if (!row_ok) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gc = n0 + c0 + 8 * h;               // the same for every lane: the routing below is warp-uniform
      if (gc >= p.N_out) break;
      uint4 v;
      v.x = pack_bf16(__uint_as_float(r[8 * h + 0]), __uint_as_float(r[8 * h + 1]));
      v.y = pack_bf16(__uint_as_float(r[8 * h + 2]), __uint_as_float(r[8 * h + 3]));
      v.z = pack_bf16(__uint_as_float(r[8 * h + 4]), __uint_as_float(r[8 * h + 5]));
      v.w = pack_bf16(__uint_as_float(r[8 * h + 6]), __uint_as_float(r[8 * h + 7]));
      if (p.mode == 1 || (p.mode == 2 && gc < 2 * w)) {
        const bool is_v = gc >= w;
        const int cc = is_v ? gc - w : gc;
        const int g = cc >> hs, c = cc & (p.hd - 1);
        __nv_bfloat16* dst = (is_v ? p.base_v : p.base_k) + base_row + ((long long)(g * PAGE) << hs) + c;
        *reinterpret_cast<uint4*>(dst) = v;
      } else {
        const int gl = p.mode == 2 ? gc - 2 * w : gc;
        const bool is_v = gl >= n_lrk;
        const int sh = is_v ? p.rv_shift : p.rk_shift;
        const int cc = is_v ? gl - n_lrk : gl;
        const int agent = cc >> sh, ri = cc & ((1 << sh) - 1);
        if (!((row_mask >> agent) & 1ull)) continue;
        __nv_bfloat16* arr = (is_v ? p.lr_v : p.lr_k) + (((long long)agent * p.n_blocks * PAGE) << sh) + ri;
        *reinterpret_cast<uint4*>(arr + (slot << sh)) = v;
        if (slot2 >= 0) *reinterpret_cast<uint4*>(arr + (slot2 << sh)) = v;
      }
    }
  }
}

__global__ void __launch_bounds__(GEMM_THREADS, 1)
proj_gemm_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const GemmParams p) {
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment for the 128-byte swizzle atoms
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int b_bytes = p.BN * GEMM_BK * 2;
  const int stage_bytes = GEMM_A_BYTES + b_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)p.stages * stage_bytes);
  // barrier map: full[stages] | empty[stages] | acc_full[2] | acc_empty[2]
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * p.stages;
  const uint32_t acc_full = empty0 + 8 * p.stages;
  const uint32_t acc_empty = acc_full + 16;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * p.stages + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = p.K / GEMM_BK;
  const int n_tiles_n = (p.N_out + p.BN - 1) / p.BN;
  // Row tiles.  With a single column tile the kernel is HBM-bound on X, and a row-tile count that is not a
  // multiple of the grid leaves part of the machine idle in the last round (256 tiles on 148 blocks = 1.73
  // rounds).  Then the count is rounded up to a multiple of the grid and the tiles are spread evenly over
  // the rows: neighbours overlap by a few rows, which are computed twice with identical results (the
  // overlap is re-read from L2, not from DRAM), and every block streams the same number of rows.
  const int m_plain = (p.M + GEMM_BM - 1) / GEMM_BM;
  const bool spread = n_tiles_n == 1 && m_plain > (int)gridDim.x && p.M >= GEMM_BM;
  const int m_tiles = spread ? ((m_plain + (int)gridDim.x - 1) / (int)gridDim.x) * (int)gridDim.x : m_plain;
  const int n_tiles = m_tiles * n_tiles_n;
  auto row0_of = [&](int mt) -> int {
    if (!spread) return mt * GEMM_BM;
    return (int)(((long long)mt * (p.M - GEMM_BM)) / (m_tiles - 1));   // first tile at 0, last one ends at M
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    mbar_init(acc_full, 1); mbar_init(acc_full + 8, 1);
    mbar_init(acc_empty, 4); mbar_init(acc_empty + 8, 4);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_holder)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  // The set-up above overlaps the end of the kernel ahead (programmatic dependent launch).  Everything that kernel may have
  // written comes after the wait, the packed weights included: its writes are visible only then.
  pdl_wait();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem_base = *tmem_holder;

  // Persistent: this block takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...; the column tile index
  // runs fastest, so blocks working at the same time share their row tile of X in L2.  The shared
  // memory ring runs straight through tile boundaries and the accumulator is double-buffered in TMEM,
  // so the epilogue of one tile overlaps the MMAs of the next.
  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int m0 = row0_of(t / n_tiles_n), n0 = (t % n_tiles_n) * p.BN;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % p.stages;
          if (it >= p.stages) mbar_wait(empty0 + 8 * s, ((it / p.stages) - 1) & 1, p.status);
          GEMM_STAMP(p, it, 0);
          const uint32_t sa = smem_u32(smem + (size_t)s * stage_bytes);
          mbar_expect_tx(full0 + 8 * s, stage_bytes);
          tma_load_2d(sa, &map_x, kb * GEMM_BK, m0, full0 + 8 * s);
          tma_load_3d(sa + GEMM_A_BYTES, &map_w, 0, n0, kb, full0 + 8 * s);      // packed weights are k-blocked
          GEMM_STAMP(p, it, 1);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(p.BN);
      const uint64_t da0 = umma_desc_sw128(smem_u32(smem));
      const uint64_t db0 = umma_desc_sw128(smem_u32(smem) + GEMM_A_BYTES);
      int it = 0, i = 0;
      for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
        const int buf = i & 1;
        if (i >= 2) mbar_wait(acc_empty + 8 * buf, ((i >> 1) - 1) & 1, p.status);   // epilogue has drained this buffer
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t d = tmem_base + buf * p.BN;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % p.stages;
          mbar_wait(full0 + 8 * s, (it / p.stages) & 1, p.status);
          GEMM_STAMP(p, it, 2);
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint64_t so = (uint64_t)((s * stage_bytes) >> 4);
#pragma unroll
          for (int k = 0; k < GEMM_BK / 16; ++k)   // 16 bf16 = 32 bytes = 2 descriptor units per step
            umma_bf16(d, da0 + so + 2 * k, db0 + so + 2 * k, idesc, (kb | k) ? 1u : 0u);
          GEMM_STAMP(p, it, 3);
          umma_commit(empty0 + 8 * s);             // stage reusable once these MMAs have read it
          GEMM_STAMP(p, it, 4);
        }
        umma_commit(acc_full + 8 * buf);           // accumulator of this tile complete
      }
    }
  } else {
    // ---- epilogue: TMEM lane = tile row; this warp may touch lanes 32*(warp%4) .. +31
    const int lane_base = (warp & 3) * 32;
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      const int buf = i & 1;
      const int m0 = row0_of(t / n_tiles_n), n0 = (t % n_tiles_n) * p.BN;
      gemm_epilogue_tile(p, tmem_base + buf * p.BN, m0, n0, lane_base, lane, acc_full + 8 * buf, (i >> 1) & 1);
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(acc_empty + 8 * buf) : "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// position of a row in the rotary table, or -1 (reported) when it is outside
__device__ __forceinline__ long long rope_pos(const GemmParams& p, int gm) {
  const long long pos = p.positions ? (long long)p.positions[gm] : p.start_pos + gm;
  if (pos >= 0 && pos < p.max_pos) return pos;
  atomicOr(p.status, StatusBits::BAD_INDEX);
  return -1;
}

}  // namespace precc
