// Projection for a handful of rows (decode steps, M <= 64): Y[M x n_out] = X[M x K] . Wt^T with the same
// routing epilogue as the tensor-memory GEMM (LR caches, base caches, or both).
//
// With M this small the work is one pass over the packed weights (n_out x K bf16), so the kernel is a
// weight-streaming kernel: HBM-bound at n_out*K*2 bytes.  A 128-row tcgen05 tile would leave all but
// n_out/BN blocks idle; here the grid covers every SM:
//   block  = 64 output columns (128 when M > 16) x one K slice; the K slices of a column group form a
//            thread-block cluster (split-K, up to 8);
//   loads  = TMA: per 64-deep k step one box of W rows (contiguous in memory: the packed weights are
//            k-blocked, [K/64][n_out][64]) and one box of X rows (rows past M are zero-filled
//            by the out-of-bounds rule) into a ring of 3 or 4 slots of 128-byte-swizzled shared memory, issued by
//            a producer warp (full/empty mbarriers).  The ring is kept small on purpose: every cluster of
//            the grid must be resident at once, or the launch runs in two waves;
//   math   = mma.sync m16n8k16 (bf16 -> fp32): X rows on the M axis, a warp owns 8 (16 when M > 16)
//            output columns; fragments come from shared memory with ldmatrix;
//   reduce = every block finishes a share of its group's tile: a slice of the columns, or (`by_rows`) some rows, all
//            columns of them.  The consumer threads SEND their accumulator pairs to the block that owns them (st.async into the owner's
//            shared memory, bytes counted on the owner's mbarrier); the owner waits for its byte count, adds the
//            partials in rank order (deterministic) and scatters bf16 pieces into the paged caches.  No global scratch, no
//            atomics, and no cluster barrier on the critical path (one, relaxed, at the start makes the mbarriers visible).
// Rotary keys (GemmParams::rope) need `by_rows`: the thread of a piece of the lower half of a head also adds up the partner piece
// hd/2 columns further, which is in the same row, and writes both rotated; the block tile holds whole heads.  (With columns
// owned by blocks the halves of a head met through a cluster barrier and loads over distributed shared memory: 3584 -> 1280
// columns, 1 / 16 / 40 rows 8.1 / 9.0 / 9.9 us, now 5.4 / 6.0 / 7.7.)  Without rotation shares of columns are the cheaper ones to send
// from eight rows on (4096 -> 2304, 16 / 32 rows: 6.1 / 7.8 us against 6.6 / 9.1: a warp's pairs then go to one block instead of
// eight).  For up to four rows, where the grid puts more than one block on an SM, rows win: most blocks own nothing and leave
// at once, which makes room for the kernel behind (one row 5.95 -> 5.70 us; 8 layers of a two-row step with their
// attention 135.8 -> 129.8).  With one block per SM it does not (2048 -> 1152: 3.05 against 3.12).
// The K split depends on K alone, so an output value does not depend on which entry point, which other
// columns or how many other rows were in the call.
#pragma once
#include "gemm_tc.cuh"

namespace precc {

constexpr int PS_WARPS = 8;
constexpr int PS_BK = 64;                   // k elements per step: one 128-byte swizzle row
constexpr int PS_THREADS = (PS_WARPS + 1) * 32;       // consumer warps + one producer warp
// Ring depth.  Above 32 rows three slots: with four (130 KB a block) only 15 clusters of eight are resident at once and the
// 18 of the Llama-3-8B projection ran in two waves (33 .. 40 rows: 12.8 us, now 9.7).
__host__ __device__ constexpr int ps_stages(int mt) { return mt > 2 ? 3 : 4; }
__host__ __device__ constexpr int ps_nt(int mt) { return mt > 1 ? 2 : 1; }               // 8-column n-tiles per warp
__host__ __device__ constexpr int ps_cols(int mt) { return PS_WARPS * 8 * ps_nt(mt); }   // output columns per block
__host__ __device__ constexpr int ps_step_bytes(int mt) { return (ps_cols(mt) + mt * 16) * PS_BK * 2; }
__host__ __device__ constexpr int ps_recv_bytes(int mt) { return mt * 16 * ps_cols(mt) * 4; }   // [cluster rank][row][own columns] fp32
__host__ __device__ constexpr int ps_smem_bytes(int mt) {
  return ps_stages(mt) * ps_step_bytes(mt) + 128 + ps_recv_bytes(mt) + 1024;   // ring | mbarriers | receive area | alignment slack
}

template <int MT>
__global__ void __launch_bounds__(PS_THREADS)
proj_small_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const GemmParams p,
                  const int k_slice) {
  constexpr int NT = ps_nt(MT);
  constexpr int COLS = ps_cols(MT);
  constexpr int W_BYTES = COLS * PS_BK * 2;
  constexpr int STEP_BYTES = ps_step_bytes(MT);
  constexpr int STAGES = ps_stages(MT);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint32_t rank, CS;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;\n" : "=r"(CS));
  const int group = blockIdx.x / CS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = rank * k_slice;
  const int steps = k_slice / PS_BK;
  const uint32_t tiles = smem_u32(smem);
  const uint32_t full0 = tiles + STAGES * STEP_BYTES, empty0 = full0 + 8 * STAGES;
  const uint32_t recv_bar = empty0 + 8 * STAGES;
  const uint32_t recv_u32 = full0 + 128;                // behind the barriers; never overlaid: peers send while this block computes
  const bool by_rows = p.by_rows != 0;                  // the same in every block of the grid
  const int cpb = COLS / CS;                            // columns finished by one block (a power of two >= 8)
  const int tw = (p.M + (int)CS - 1) / (int)CS;         // by rows: rows finished by one block (the last ones may own fewer, or none)
  const int own = max(0, min(tw, p.M - (int)rank * tw));

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, PS_WARPS); }
    mbar_init(recv_bar, 1);
    // the one arrival, and the bytes to come: the own rows of every peer, or rows < M of the own columns
    mbar_expect_tx(recv_bar, by_rows ? (uint32_t)((int)CS * own * COLS * 4) : (uint32_t)(CS * p.M * cpb * 4));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");   // waited for before the first send
  // The weights are not the preceding kernel's to write: the first ring fill of W boxes is requested before the wait
  // for that kernel (programmatic dependent launch), so a block that is resident early has them in shared memory
  // when its predecessor ends.  X (the previous kernel's output) and every store stay behind the wait.
  const int pre = steps < STAGES ? steps : STAGES;
  if (warp == PS_WARPS && lane == 0) {
    for (int s = 0; s < pre; ++s) {
      mbar_expect_tx(full0 + 8 * s, STEP_BYTES);
      tma_load_3d(tiles + s * STEP_BYTES, &map_w, 0, group * COLS, k0 / PS_BK + s, full0 + 8 * s);
    }
  }
  pdl_wait();                 // X may be the previous kernel's output; the caches may still be read by it
  pdl_launch_dependents();

  float acc[MT][NT][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int t = 0; t < NT; ++t) { acc[mt][t][0] = acc[mt][t][1] = acc[mt][t][2] = acc[mt][t][3] = 0.f; }

  if (warp == PS_WARPS) {
    // ---- producer: one lane walks the k steps of this block's slice
    if (lane == 0) {
      for (int s = 0; s < pre; ++s)                      // the X boxes of the steps whose W boxes are already on their way
        tma_load_2d(tiles + s * STEP_BYTES + W_BYTES, &map_x, k0 + s * PS_BK, 0, full0 + 8 * s);
      for (int s = pre; s < steps; ++s) {
        const int slot = s % STAGES;
        mbar_wait(empty0 + 8 * slot, ((s / STAGES) - 1) & 1, p.status);
        const uint32_t dst = tiles + slot * STEP_BYTES;
        mbar_expect_tx(full0 + 8 * slot, STEP_BYTES);
        tma_load_3d(dst, &map_w, 0, group * COLS, k0 / PS_BK + s, full0 + 8 * slot);   // one contiguous run of the k-blocked weights
        tma_load_2d(dst + W_BYTES, &map_x, k0 + s * PS_BK, 0, full0 + 8 * slot);
      }
    }
  } else {
    const int mi = lane >> 3, ri = lane & 7;
    for (int s = 0; s < steps; ++s) {
      const int slot = s % STAGES;
      mbar_wait(full0 + 8 * slot, (s / STAGES) & 1, p.status);
      const uint32_t wt = tiles + slot * STEP_BYTES, xt = wt + W_BYTES;
#pragma unroll
      for (int j = 0; j < 2; ++j) {                      // two k steps of 16 per ldmatrix of W
        uint32_t b[NT][4];
#pragma unroll
        for (int t = 0; t < NT; ++t) ldsm_x4(b[t], wt + swz_off<8>((warp * NT + t) * 8 + ri, 4 * j + mi));
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t a[4];
            ldsm_x4(a, xt + swz_off<8>(mt * 16 + ri + (mi & 1) * 8, 2 * (2 * j + h) + (mi >> 1)));
#pragma unroll
            for (int t = 0; t < NT; ++t) mma_bf16_16816(acc[mt][t], a, b[t][2 * h], b[t][2 * h + 1]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(empty0 + 8 * slot) : "memory");
    }
  }
  if (!by_rows) {
    // ---- merge by sends: accumulator pairs go straight from registers to the owner of their column
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");   // every peer's mbarrier is initialised (long since)
    const int cshift = 31 - __clz(cpb);
    if (warp < PS_WARPS) {
      const int r = lane >> 2, q = lane & 3;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const int col = (warp * NT + t) * 8 + 2 * q;
          const int owner = col >> cshift;
          const uint32_t bar = dsmem_addr(recv_bar, owner);
          const uint32_t dst = recv_u32 + (uint32_t)(((rank * (MT * 16) + mt * 16 + r) * cpb + (col & (cpb - 1))) * 4);
          if (mt * 16 + r < p.M) st_async_f32x2(dsmem_addr(dst, owner), acc[mt][t][0], acc[mt][t][1], bar);
          if (mt * 16 + r + 8 < p.M) st_async_f32x2(dsmem_addr(dst + 8 * cpb * 4, owner), acc[mt][t][2], acc[mt][t][3], bar);
        }
    }
    // ---- this block finishes columns [rank*cpb, (rank+1)*cpb) of its group: 8-column pieces, partials added in rank order
    const int ppr = cpb / 8;
    const int n_items = p.M * ppr;
    int it = threadIdx.x;
    int row = it / ppr, pc = it - row * ppr;              // worked out before the wait
    mbar_wait_cluster(recv_bar, 0, p.status);
    const float* recv = reinterpret_cast<const float*>(smem + STAGES * STEP_BYTES + 128);
    for (; it < n_items; it += PS_THREADS, row = it / ppr, pc = it - row * ppr) {
      const int gc = group * COLS + rank * cpb + pc * 8;
      if (gc >= p.N_out) continue;
      long long slot = p.slot_mapping ? (long long)p.slot_mapping[row] : p.start_slot + row;
      if (slot < 0 || slot >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); continue; }
      const unsigned long long mask = p.row_masks ? p.row_masks[row] : p.agent_mask;
      float4 x0[8], x1[8];
#pragma unroll
      for (uint32_t s = 0; s < 8; ++s) {
        if (s < CS) {
          const float* src = recv + ((size_t)(s * (MT * 16) + row) * cpb + pc * 8);
          x0[s] = *reinterpret_cast<const float4*>(src);
          x1[s] = *reinterpret_cast<const float4*>(src + 4);
        } else {
          x0[s] = make_float4(0.f, 0.f, 0.f, 0.f); x1[s] = x0[s];
        }
      }
      float v8[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v8[k] = 0.f;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        v8[0] += x0[s].x; v8[1] += x0[s].y; v8[2] += x0[s].z; v8[3] += x0[s].w;
        v8[4] += x1[s].x; v8[5] += x1[s].y; v8[6] += x1[s].z; v8[7] += x1[s].w;
      }
      store_piece(p, slot / PAGE, (int)(slot % PAGE), gc, v8, mask, row);
    }
    return;     // a block leaves once everything addressed to it has arrived; its own sends carry their data with them
  }
  // ---- the same with rows: pairs go to the owner of their row, which has all columns of it
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  if (warp < PS_WARPS) {
    const int r = lane >> 2, q = lane & 3;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = mt * 16 + 8 * h + r;
        if (row >= p.M) continue;
        const int owner = row / tw;
        const uint32_t bar = dsmem_addr(recv_bar, owner);
        const uint32_t dst = dsmem_addr(recv_u32 + (uint32_t)((((int)rank * tw + row - owner * tw) * COLS + warp * NT * 8 + 2 * q) * 4), owner);
#pragma unroll
        for (int t = 0; t < NT; ++t) st_async_f32x2(dst + t * 32, acc[mt][t][2 * h], acc[mt][t][2 * h + 1], bar);
      }
  }
  constexpr int PPR = COLS / 8;
  const int n_items = own * PPR;
  const int kw = (p.rope && p.mode != 0) ? p.n_kv * p.hd : 0;   // width of the key columns that get rotated
  const float* recv = reinterpret_cast<const float*>(smem + STAGES * STEP_BYTES + 128);
  auto gather = [&](int lr, int col, float (&v8)[8]) {          // columns [col, col + 8) of own row lr, summed over the cluster in rank order
    float4 x0[8], x1[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      if (s < (int)CS) {
        const float* src = recv + (size_t)(s * tw + lr) * COLS + col;
        x0[s] = *reinterpret_cast<const float4*>(src);
        x1[s] = *reinterpret_cast<const float4*>(src + 4);
      } else {
        x0[s] = make_float4(0.f, 0.f, 0.f, 0.f); x1[s] = x0[s];
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) v8[k] = 0.f;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      v8[0] += x0[s].x; v8[1] += x0[s].y; v8[2] += x0[s].z; v8[3] += x0[s].w;
      v8[4] += x1[s].x; v8[5] += x1[s].y; v8[6] += x1[s].z; v8[7] += x1[s].w;
    }
  };
  mbar_wait_cluster(recv_bar, 0, p.status);
  for (int it = threadIdx.x; it < n_items; it += PS_THREADS) {
    const int lr = it / PPR, col = (it % PPR) * 8, row = (int)rank * tw + lr;
    const int gc = group * COLS + col;
    if (gc >= p.N_out) continue;
    if (gc < kw && (gc & (p.hd - 1)) >= p.hd / 2) continue;   // upper half of a rotated head: written with its lower partner
    const long long slot = p.slot_mapping ? (long long)p.slot_mapping[row] : p.start_slot + row;
    if (slot < 0 || slot >= p.n_blocks * PAGE) { atomicOr(p.status, StatusBits::BAD_INDEX); continue; }
    const unsigned long long mask = p.row_masks ? p.row_masks[row] : p.agent_mask;
    float v8[8];
    gather(lr, col, v8);
    if (gc < kw) {
      const long long pos = rope_pos(p, row);
      if (pos < 0) continue;
      float h8[8];
      gather(lr, col + p.hd / 2, h8);
      const float4* cs = p.rope + pos * (p.hd / 4) + (gc & (p.hd - 1)) / 2;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 t4 = __ldg(cs + k);                // (cos c, sin c, cos c+1, sin c+1)
        const float l0 = v8[2 * k], l1 = v8[2 * k + 1], h0 = h8[2 * k], h1 = h8[2 * k + 1];
        v8[2 * k] = l0 * t4.x - h0 * t4.y; v8[2 * k + 1] = l1 * t4.z - h1 * t4.w;
        h8[2 * k] = h0 * t4.x + l0 * t4.y; h8[2 * k + 1] = h1 * t4.z + l1 * t4.w;
      }
      store_piece(p, slot / PAGE, (int)(slot % PAGE), gc + p.hd / 2, h8, mask, row);
    }
    store_piece(p, slot / PAGE, (int)(slot % PAGE), gc, v8, mask, row);
  }
}

}  // namespace precc
