// Adapted rotary keys of one sequence, written out once for a turn's prefill (Appendix D.2: the key-side adapter
// term sits inside the rotation, so it cannot be folded into the query).  For every token t of the sequence,
// kv head g and column pair (c, c + hd/2):
//     K_a[t][g][:] = K_base_rot[t][g][:] + s_k RoPE_t( L^K_a[t][:] B^K_a[:, g] )
// with K_base_rot the cache's (already rotated) base keys, L^K the agent's unrotated LR rows and token t at
// position t.  The result goes to a caller-provided scratch area in LOGICAL block order, layout
// [block][kv head][16][hd] like the cache, so that the tensor-memory prefill kernel can stream it as its key
// operand with whole-stage boxes and no key-side adapter at all.
#pragma once
#include "common.cuh"

namespace precc {

struct RopeExpandParams {
  const __nv_bfloat16* k_base;   // [n_blocks][n_kv][16][hd]
  const __nv_bfloat16* lr_k;     // the agent's rows: [n_blocks][16][rk]
  const __nv_bfloat16* B_k;      // the agent's matrix: [rk][n_kv * hd]
  const float4* rope;            // [max_pos][hd/4] of (cos c, sin c, cos c+1, sin c+1), c even
  const int32_t* block_table;    // logical -> physical block, or null
  __nv_bfloat16* scratch;        // [n_out_blocks][n_kv][16][hd]
  uint32_t* status;
  long long n_blocks;            // physical blocks of the cache
  int first_block;               // physical block of logical block 0 when block_table is null
  int n_tokens;                  // tokens of the sequence (context + turn); rows past it are written as zeros
  int n_out_blocks;              // cache blocks to write (whole 128-token stages)
  int n_kv, hd, rk, max_pos;
  float s_k;
};

// E = L^K B^K on the tensor cores (mma.sync m16n8k16: the 16 tokens of a cache block on the M axis, rank on K, columns
// on N).  A warp owns 32 columns of the lower half of one head and their partners in the upper half: eight n-tiles, whose
// columns are handed out so that a lane ends up with EIGHT ADJACENT columns of its two tokens in either half (n-tile t,
// column n of it = column 8 (n / 2) + 2 t + (n & 1) of the 32): base keys, scratch and rotary table are then read and
// written with 16-byte accesses straight from and to the accumulator layout, and nothing passes through shared memory.
// A warp keeps its B^K fragments in registers and walks over cache blocks; warps know nothing of each other.
// (The term used to be parked in shared memory between two block barriers per cache block: a call of 32 new tokens over 8000 with 4 kv
// heads of 128, rank 16, took 32.1 us and takes 28.8; over 32768 with 8 kv heads, rank 32: 105 -> 85; head_dim 64, rank 64, 16000: 53 -> 41.)
// KS = k steps of 16 (rank 8 and 16: 1, rank 32: 2, rank 64: 4).
constexpr int RX_WARPS = 4;
constexpr int RX_THREADS = RX_WARPS * 32;
constexpr int RX_COLS = 64;                              // columns of a warp: 32 of the lower half of a head, 32 of the upper

__host__ __device__ constexpr int rx_blocks_per_sm(int ks) { return ks == 4 ? 2 : ks == 2 ? 3 : 4; }   // what the registers allow

template <int KS>
__global__ void __launch_bounds__(RX_THREADS, rx_blocks_per_sm(KS))
rope_expand_keys_kernel(const RopeExpandParams p) {
  const int hd = p.hd, rk = p.rk;
  const int kvw = p.n_kv * hd;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane >> 2, q = lane & 3;                 // accumulator rows (tokens) r, r + 8; columns 8 q .. 8 q + 7 of either half
  const int per_head = hd / RX_COLS;
  const int task = blockIdx.y * RX_WARPS + warp;
  if (task >= p.n_kv * per_head) return;
  const int g = task / per_head, c0 = (task - g * per_head) * 32;      // head, first column in its lower half
  pdl_wait();                  // the kernel ahead may have written anything that is read below
  int lb = blockIdx.x;
  auto lookup = [&](int b) -> int {
    if (b * PAGE >= p.n_tokens) return 0;
    const int ph = p.block_table ? __ldg(p.block_table + b) : p.first_block + b;
    if (ph >= 0 && ph < p.n_blocks) return ph;
    if (lane == 0 && task == 0) atomicOr(p.status, StatusBits::BAD_INDEX);
    return 0;
  };
  // ---- inputs of one cache block, requested a block ahead of their use (its place in the cache two ahead): base keys of
  //      the lane's two tokens in both halves and L^K rows r, r + 8, zero past the sequence's end
  struct In { uint4 kb[2][2]; uint32_t afr[KS][4]; };
  auto fetch = [&](int b, int ph, In& x) {
    const int t0 = b * PAGE;
    const bool any = t0 < p.n_tokens;
    const __nv_bfloat16* src = p.k_base + ((size_t)((size_t)ph * p.n_kv + g) * PAGE + r) * hd + c0 + q * 8;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool on = t0 + r + 8 * h < p.n_tokens;
      x.kb[h][0] = on ? __ldg(reinterpret_cast<const uint4*>(src + h * 8 * hd)) : make_uint4(0u, 0u, 0u, 0u);
      x.kb[h][1] = on ? __ldg(reinterpret_cast<const uint4*>(src + h * 8 * hd + hd / 2)) : make_uint4(0u, 0u, 0u, 0u);
    }
    const __nv_bfloat16* lrow = p.lr_k + ((size_t)ph * PAGE + r) * rk;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      const int k = ks * 16 + q * 2;
      x.afr[ks][0] = any && k < rk ? __ldg(reinterpret_cast<const uint32_t*>(lrow + k)) : 0u;
      x.afr[ks][1] = any && k < rk ? __ldg(reinterpret_cast<const uint32_t*>(lrow + 8 * rk + k)) : 0u;
      x.afr[ks][2] = any && k + 8 < rk ? __ldg(reinterpret_cast<const uint32_t*>(lrow + k + 8)) : 0u;
      x.afr[ks][3] = any && k + 8 < rk ? __ldg(reinterpret_cast<const uint32_t*>(lrow + 8 * rk + k + 8)) : 0u;
    }
  };
  if (lb >= p.n_out_blocks) return;
  In cur;
  fetch(lb, lookup(lb), cur);
  int ph_next = lb + (int)gridDim.x < p.n_out_blocks ? lookup(lb + gridDim.x) : 0;
  // ---- B^K fragments (k = rank, n = column), zero beyond the rank; tiles 0 .. 3 lower half, 4 .. 7 upper
  uint32_t bfr[8][KS][2];
  {
    const unsigned short* B = reinterpret_cast<const unsigned short*>(p.B_k) + (size_t)g * hd + c0 + (r >> 1) * 8 + (r & 1);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const unsigned short* Bt = B + (t & 3) * 2 + (t >> 2) * (hd / 2);
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int k0 = ks * 16 + q * 2;
        auto bk = [&](int k) -> uint32_t { return k < rk ? (uint32_t)__ldg(Bt + (size_t)k * kvw) : 0u; };
        bfr[t][ks][0] = bk(k0) | (bk(k0 + 1) << 16);
        bfr[t][ks][1] = bk(k0 + 8) | (bk(k0 + 9) << 16);
      }
    }
  }
  for (; lb < p.n_out_blocks; lb += gridDim.x) {
    const int t0 = lb * PAGE, nb = lb + gridDim.x;
    In nxt = cur;
    if (nb < p.n_out_blocks) {
      fetch(nb, ph_next, nxt);
      if (nb + (int)gridDim.x < p.n_out_blocks) ph_next = lookup(nb + gridDim.x);
    }
    __nv_bfloat16* dst = p.scratch + ((size_t)((size_t)lb * p.n_kv + g) * PAGE + r) * hd + c0 + q * 8;
    float4 cs[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4* cs4 = p.rope + (size_t)min(t0 + r + 8 * h, p.max_pos - 1) * (hd / 4) + (c0 + q * 8) / 2;
#pragma unroll
      for (int t = 0; t < 4; ++t) cs[h][t] = __ldg(cs4 + t);
    }
    float acc[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) mma_bf16_16816(acc[t], cur.afr[ks], bfr[t][ks][0], bfr[t][ks][1]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t lo[4], hi[4];
      const uint32_t kl[4] = {cur.kb[h][0].x, cur.kb[h][0].y, cur.kb[h][0].z, cur.kb[h][0].w};
      const uint32_t kh[4] = {cur.kb[h][1].x, cur.kb[h][1].y, cur.kb[h][1].z, cur.kb[h][1].w};
      auto add2 = [](uint32_t k2, float a, float b) -> uint32_t {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&k2));
        return pack_bf16(f.x + a, f.y + b);
      };
#pragma unroll
      for (int t = 0; t < 4; ++t) {                      // columns 2 t, 2 t + 1 of the lane's eight
        const float4 c4 = cs[h][t];
        const float lo0 = p.s_k * acc[t][2 * h], lo1 = p.s_k * acc[t][2 * h + 1];
        const float hi0 = p.s_k * acc[t + 4][2 * h], hi1 = p.s_k * acc[t + 4][2 * h + 1];
        lo[t] = add2(kl[t], lo0 * c4.x - hi0 * c4.y, lo1 * c4.z - hi1 * c4.w);
        hi[t] = add2(kh[t], hi0 * c4.x + lo0 * c4.y, hi1 * c4.z + lo1 * c4.w);
      }
      const bool on = t0 + r + 8 * h < p.n_tokens;       // rows past the sequence's end, and the padding up to a whole 128-token stage: zeros
      *reinterpret_cast<uint4*>(dst + h * 8 * hd) = on ? make_uint4(lo[0], lo[1], lo[2], lo[3]) : make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(dst + h * 8 * hd + hd / 2) = on ? make_uint4(hi[0], hi[1], hi[2], hi[3]) : make_uint4(0u, 0u, 0u, 0u);
    }
    cur = nxt;
  }
}

}  // namespace precc
