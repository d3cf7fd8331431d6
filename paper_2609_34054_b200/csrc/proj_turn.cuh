// Projection for the tokens of a turn (about 40 .. 2000 rows): Y[M x n_out] = X[M x K] . Wt^T with the routing of the
// other projection kernels (LR caches, base caches, or both).
//
// With this few rows the launch is bound by what a block takes in per k-block (about 0.37 us each) and by what it costs to
// add up the K slices, so both are kept small:
//   tile   = 128 output columns x TN rows (TN <= 256, a multiple of 16).  The WEIGHTS are the M = 128 operand of
//            tcgen05.mma and the rows of X its N operand: a tile is as wide as there are rows, instead of 128-row
//            steps of padding, and a block takes in (128 + TN) x 128 bytes per k-block;
//   split  = the K extent of a tile over the KS blocks of a cluster (1 .. 8; K slices need not be equal);
//   merge  = block r finishes ROWS [r tw, (r+1) tw) of the tile, all 128 columns of them.  Tensor memory holds a column
//            of the output per lane, so the dump to shared memory is one conflict-free 4-byte store per row and
//            lane, and a row of the dump is 128 consecutive columns: the slice for block j is ONE run of memory,
//            sent with one cp.async.bulk (shared::cta -> shared::cluster, bytes counted on an mbarrier of the receiver)
//            while the next slice is dumped.  The receiver adds the KS slices in rank order (the result does not
//            depend on timing) and stores 16-byte pieces, sixteen lanes on consecutive pieces of a row.  Whole heads sit in
//            one row of the tile, so rotary keys find their partner column next to them.
// NG = 2: one block takes 256 columns of its rows (two accumulators of up to 256 tensor-memory columns), KS = 1.  This is the
// form for many rows and few columns (the LR rows of a long context), which is bound by the rows of X: cut into as many tiles
// as there are SMs, every row is fetched once and the weights once per SM, where 128-row tiles come out as two rounds of
// overlapping ones (32768 rows x 256 columns of d_model 4096: 71.5 -> 64.0 us; 20000 x 192: 56.6 -> 42.1; 20000 x 128, NG = 1: 53.0 -> 35.9).
// Shared memory: [ring of {W 128 NG x 64 | X TN x 64} | overlaid: dump [TN][128] fp32, receive area [KS-1][tw][128] fp32]
// [row table][barriers].  A block tells its peers when its ring is idle; they send only then.
// The K split depends on M, K and the layer's fused width alone, so base-only, LR-only and fused calls agree bit for bit; TN, which changes no bit,
// on the columns of the call (proj_plan.h).
// Measured on rotating weights from HBM, us a launch, against 128-row x 256-column tiles whose slices were pulled over
// distributed shared memory (or sent, clusters of up to four) with 128 threads: 4096 -> 2304 columns, 64 / 128 / 301 / 512 / 1024 rows:
// 12.4 / 15.1 / 16.6 / 19.5 / 24.5 -> 10.1 / 11.3 / 15.3 / 17.2 / 20.9; 2048 -> 1152: 9.8 / 12.7 / 13.2 / 14.7 / 15.3 -> 7.5 / 7.8 / 9.1 /
// 10.3 / 12.5; 3584 -> 1280 with rotary keys, 64 / 200 / 512: 11.6 / 15.7 / 18.4 -> 9.1 / 10.9 / 13.6; 1024 -> 560: 8.6 .. 13.8 -> 5.8 .. 8.5.
// (Up to 64 rows the three narrower layers run on the few-row kernel, see few_row_limit.)
#pragma once
#include "gemm_tc.cuh"

namespace precc {

constexpr int PT_EPI_WARPS = 8;
constexpr int PT_THREADS = (2 + PT_EPI_WARPS) * 32;      // producer, MMA issuer, eight merging warps

template <bool ROPE, int NG>
__global__ void __launch_bounds__(PT_THREADS, 1)
proj_turn_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const GemmParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw;
  if ((smem_u32(smem_raw) & 1023u) != 0) {               // the swizzle atoms and the peers' addresses rely on it
    if (threadIdx.x == 0) atomicOr(p.status, StatusBits::TIMEOUT);
    return;
  }
  const int KS = gridDim.x, rank = blockIdx.x;           // the cluster spans grid.x
  const int TN = p.BN;
  const int stage_bytes = pt_stage_bytes(TN, NG);
  PtRow* rows = reinterpret_cast<PtRow*>(smem + pt_data_bytes(TN, KS, p.stages, NG));
  uint64_t* bars = reinterpret_cast<uint64_t*>(rows + pt_share(TN, KS));
  // barrier map: full[stages] | empty[stages] | acc_full | ready (peers whose ring is idle) | recv (bytes received)
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * PT_MAX_STAGES;
  const uint32_t acc_full = empty0 + 8 * PT_MAX_STAGES;
  const uint32_t ready_bar = acc_full + 8, recv_bar = acc_full + 16;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * PT_MAX_STAGES + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = p.K / GEMM_BK;
  const int kb0 = (rank * nkb) / KS;
  const int nkb_s = ((rank + 1) * nkb) / KS - kb0;
  const int m0 = blockIdx.z * TN, n0 = blockIdx.y * (NG * PT_COLS);
  const int n_rows = min(TN, p.M - m0);                  // rows of this tile that exist
  const int tw = pt_share(n_rows, KS);                   // rows finished by one block (the last ones may own fewer, or none)
  auto slice_rows = [&](int r) { return max(0, min(tw, n_rows - r * tw)); };
  const int own_rows = slice_rows(rank);
  float* dump = reinterpret_cast<float*>(smem);                               // [n_rows][128]
  float* recv = dump + (size_t)TN * PT_COLS;                                  // [KS-1][tw][128], slot = sender's rank with the own rank left out

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    mbar_init(acc_full, 1);
    mbar_init(ready_bar, KS > 1 ? KS - 1 : 1);
    mbar_init(recv_bar, 1);
    mbar_expect_tx(recv_bar, (uint32_t)((KS - 1) * own_rows * PT_COLS * 4));   // the one arrival, and the bytes to come
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    // the ring's first fill is requested right behind the wait for the kernel ahead (this thread is the producer): its
    // latency then overlaps the tensor-memory allocation and the block barrier below
    pdl_wait();
    for (int it = 0; it < min(p.stages, nkb_s); ++it) {
      const uint32_t st = smem_u32(smem) + it * stage_bytes;
      mbar_expect_tx(full0 + 8 * it, stage_bytes);
      tma_load_3d(st, &map_w, 0, n0, kb0 + it, full0 + 8 * it);
      tma_load_2d(st + NG * PT_W_BYTES, &map_x, (kb0 + it) * GEMM_BK, m0, full0 + 8 * it);
    }
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_holder)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  pdl_wait();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem_base = *tmem_holder;
  // every block's barriers exist before anybody arrives on them from outside (the wait comes with the first remote use)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      for (int it = p.stages; it < nkb_s; ++it) {
        const int s = it % p.stages;
        mbar_wait(empty0 + 8 * s, ((it / p.stages) - 1) & 1, p.status);
        const uint32_t st = smem_u32(smem) + s * stage_bytes;
        mbar_expect_tx(full0 + 8 * s, stage_bytes);
        tma_load_3d(st, &map_w, 0, n0, kb0 + it, full0 + 8 * s);
        tma_load_2d(st + NG * PT_W_BYTES, &map_x, (kb0 + it) * GEMM_BK, m0, full0 + 8 * s);
      }
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(TN);
      const uint64_t dw0 = umma_desc_sw128(smem_u32(smem));
      const uint64_t dx0 = umma_desc_sw128(smem_u32(smem) + NG * PT_W_BYTES);
      for (int it = 0; it < nkb_s; ++it) {
        const int s = it % p.stages;
        mbar_wait(full0 + 8 * s, (it / p.stages) & 1, p.status);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint64_t so = (uint64_t)((s * stage_bytes) >> 4);
#pragma unroll
        for (int k = 0; k < GEMM_BK / 16; ++k)
#pragma unroll
          for (int h = 0; h < NG; ++h)
            umma_bf16(tmem_base + h * PT_MAX_TN, dw0 + so + h * (PT_W_BYTES >> 4) + 2 * k, dx0 + so + 2 * k, idesc, (it | k) ? 1u : 0u);
        umma_commit(empty0 + 8 * s);
      }
      umma_commit(acc_full);                       // every MMA of the slice has completed: the ring is idle too
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2;   // tensor-memory lanes of this warp; which of the two warps on them
    const int et = threadIdx.x - 64;                     // 0 .. 255 among the merging threads
    // ---- the routing of this block's rows and of this thread's eight columns, worked out under the main loop
    if (et < own_rows) {
      const int gm = m0 + rank * tw + et;
      PtRow r{0, -1, p.row_masks ? p.row_masks[gm] : p.agent_mask, 0, 1};
      r.slot = p.slot_mapping ? (long long)p.slot_mapping[gm] : p.start_slot + gm;
      if (r.slot < 0 || r.slot >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); r.ok = 0; r.slot = 0; }
      if (r.ok && p.lr_copy_slots) {
        r.slot2 = p.lr_copy_slots[gm];
        if (r.slot2 >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); r.slot2 = -1; }
      }
      if constexpr (ROPE) {
        if (r.ok) { const long long pos = rope_pos(p, gm); r.ok = pos >= 0; r.pos = (int)(pos >= 0 ? pos : 0); }
      }
      rows[et] = r;
    }
    const int piece = et & 15;                           // eight columns: the same ones in every pass of the reduction below
#pragma unroll 1
    for (int h = 0; h < NG; ++h) {                       // one 128-column half after the other, through the same dump
      const int gc = n0 + h * PT_COLS + piece * 8, w = p.n_kv << p.hd_shift;
      bool live = gc < p.N_out, to_base = p.mode == 1 || (p.mode == 2 && gc < 2 * w), is_key = false;
      __nv_bfloat16* dst0;                                 // base: [blk][n_kv][16][hd] at this head and column; LR: [slot][r] at this agent and coordinate
      int agent = 0, sh;                                   // sh: log2 of the destination's row width
      if (to_base) {
        const bool is_v = gc >= w;
        const int cc = is_v ? gc - w : gc;
        is_key = !is_v;
        sh = p.hd_shift;
        dst0 = (is_v ? p.base_v : p.base_k) + ((long long)((cc >> sh) * PAGE) << sh) + (cc & (p.hd - 1));
        if (ROPE && is_key && (cc & (p.hd - 1)) >= p.hd / 2) live = false;        // the upper half of a rotated head is written with the lower
      } else {
        const int n_lrk = p.rank_k > 0 ? (p.n_agents << p.rk_shift) : 0;
        const int gl = p.mode == 2 ? gc - 2 * w : gc;
        const bool is_v = gl >= n_lrk;
        sh = is_v ? p.rv_shift : p.rk_shift;
        const int cc = is_v ? gl - n_lrk : gl;
        agent = cc >> sh;
        dst0 = (is_v ? p.lr_v : p.lr_k) + (((long long)agent * p.n_blocks * PAGE) << sh) + (cc & ((1 << sh) - 1));
      }
      if (h == 0) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");       // the peers' barriers are initialised
      mbar_wait(acc_full, 0, p.status);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      // this block's ring is idle: the peers may send into the receive area that overlays it
      if (et < KS - 1) {
        const int peer = et < rank ? et : et + 1;
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(dsmem_addr(ready_bar, peer)) : "memory");
      }
      // ---- dump slice by slice, the peers' first, the own one last; a peer's slice leaves while the next is dumped
      const uint32_t trow = tmem_base + h * PT_MAX_TN + (static_cast<uint32_t>(quad * 32) << 16);
      float* dcol = dump + quad * 32 + lane;
      for (int k = 1; k <= KS; ++k) {
        const int sl = rank + k < KS ? rank + k : rank + k - KS;
        const int c0 = sl * tw, nr = slice_rows(sl);
        for (int c = half * 8; c < nr; c += 32) {          // two groups of eight rows in flight per warp (the last one may run up to seven rows past n_rows: inside the tile, never read)
          uint32_t r0[8], r1[8];
          const bool two = c + 16 < nr;
          tmem_ld8(trow + c0 + c, r0);
          if (two) tmem_ld8(trow + c0 + c + 16, r1);
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
  #pragma unroll
          for (int q = 0; q < 8; ++q)
            dcol[(size_t)(c0 + c + q) * PT_COLS] = __uint_as_float(r0[q]);
          if (two) {
  #pragma unroll
            for (int q = 0; q < 8; ++q)
              dcol[(size_t)(c0 + c + 16 + q) * PT_COLS] = __uint_as_float(r1[q]);
          }
        }
        if (k < KS) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the copy engine reads what these threads wrote
        asm volatile("bar.sync 1, 256;\n" ::: "memory");                            // the merging warps
        if (k < KS && et == 0) {
          if (k == 1) mbar_wait_cluster(ready_bar, 0, p.status);                     // every peer's ring is idle
          if (nr > 0) {
            const uint32_t src = smem_u32(dump) + (uint32_t)(c0 * PT_COLS * 4);
            const uint32_t dst = dsmem_addr(smem_u32(recv) + (uint32_t)((rank < sl ? rank : rank - 1) * tw * PT_COLS * 4), sl);
            asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                         ::"r"(dst), "r"(src), "r"(nr * PT_COLS * 4), "r"(dsmem_addr(recv_bar, sl)) : "memory");
          }
        }
      }
      // ---- own rows + received rows, in rank order, routed to the caches: sixteen threads per row, eight columns each
      mbar_wait_cluster(recv_bar, 0, p.status);
      const float* own = dump + (size_t)rank * tw * PT_COLS;
      auto gather = [&](int r, int c, float (&v)[8]) {
  #pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = 0.f;
  #pragma unroll
        for (int s = 0; s < GEMM_MAX_KS; ++s) {
          if (s < KS) {
            const float* src = (s == rank ? own : recv + (size_t)(s < rank ? s : s - 1) * tw * PT_COLS) + r * PT_COLS + c;
            const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
            v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w; v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
          }
        }
      };
      auto pack8 = [](const float (&v)[8]) {
        return make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
      };
      for (int r = et >> 4; live && r < own_rows; r += PT_EPI_WARPS * 2) {
        const PtRow row = rows[r];
        if (!row.ok) continue;
        float v[8];
        gather(r, piece * 8, v);
        if (to_base) {
          __nv_bfloat16* dst = dst0 + (((row.slot / PAGE) * p.n_kv * PAGE + (row.slot % PAGE)) << sh);
          if constexpr (ROPE) {
            if (is_key) {
              float u[8];
              gather(r, piece * 8 + p.hd / 2, u);
              const float4* cs = p.rope + (long long)row.pos * (p.hd / 4) + (gc & (p.hd - 1)) / 2;
  #pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float4 t = __ldg(cs + q);
                const float l0 = v[2 * q], l1 = v[2 * q + 1], h0 = u[2 * q], h1 = u[2 * q + 1];
                v[2 * q] = l0 * t.x - h0 * t.y; v[2 * q + 1] = l1 * t.z - h1 * t.w;
                u[2 * q] = h0 * t.x + l0 * t.y; u[2 * q + 1] = h1 * t.z + l1 * t.w;
              }
              *reinterpret_cast<uint4*>(dst + p.hd / 2) = pack8(u);
            }
          }
          *reinterpret_cast<uint4*>(dst) = pack8(v);
        } else if ((row.mask >> agent) & 1ull) {
          const uint4 o = pack8(v);
          *reinterpret_cast<uint4*>(dst0 + (row.slot << sh)) = o;
          if (row.slot2 >= 0) *reinterpret_cast<uint4*>(dst0 + (row.slot2 << sh)) = o;
        }
      }
      if (h + 1 < NG) asm volatile("bar.sync 1, 256;\n" ::: "memory");   // the dump has been read
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  }
  // the sends read the sender's shared memory: nobody leaves before every block has received everything
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

}  // namespace precc
