// Host side of decode attention: the split schedule (cluster kernel or ticket kernel), workspace sizing and
// the launch.  Included by one translation unit per head dimension.
#pragma once
#include "api_internal.h"
#include "decode.cuh"

namespace precc {

// Split schedule of decode.  cluster > 0: the cluster kernel with that many blocks per (request, kv head);
// otherwise the ticket kernel - on a flat grid of `flat` blocks, or (flat == 0) with up to max_splits blocks per (request,
// kv head).
struct DecodePlan { int cluster, warps, chunk_tiles, max_splits, stages, smem, deep, flat, even; };

template <int HD, int RK, int RV, bool ROPE = false>
struct DecodeRunT {
  // The workspace bound below is computed for the plain kernel and serves the rotary one too: the rotary blocks
  // are larger (the B_k slice rides in shared memory), which can only lower the split count - as long as two
  // of them still fit on an SM at the shallowest ring, so that the planner's blocks-per-SM figure is the same.
  static_assert(!ROPE || 2 * (DecodeCfg<HD, RK, RV>::ticket_smem(2) + DecodeCfg<HD, RK, RV>::BK_BYTES + 128 + 1024) <= 232448,
                "rotary ticket blocks must fit two per SM, or the workspace bound of the plain kernel no longer covers them");
  // Workspace: arrival counters of the (request, kv head) pairs, then records.  The counters have to be zero between calls, so
  // no call may find another one's records there: their place and size depend on the device alone, not on the batch or the
  // layer (they used to be as many as the call had pairs, and a later call of a larger batch on the same workspace took the
  // records behind them for counters: no block of such a pair saw itself as the last, and its output was never written).
  // Enough for every pair that can be split: more than one block per pair takes fewer pairs than the 4 x 2 x SMs blocks
  // that plan_split wants at most, or than the 4 x SMs of a flat grid.
  static long long counted_units(int sm_count) { return 8ll * sm_count; }
  static size_t counter_bytes(int sm_count) { return ((size_t)counted_units(sm_count) * 4 + 255) / 256 * 256; }
  // need of one call: the counters if pairs are split, and the records
  static size_t ws_need(int sm_count, bool split, long long records) {
    return (split ? counter_bytes(sm_count) : 0) + (size_t)records * DecodeCfg<HD, RK, RV>::PART_STRIDE * 4;
  }
  static int ticket_per_sm(int stages, int max_smem, int extra) {
    const int n = max_smem / (DecodeCfg<HD, RK, RV>::ticket_smem(stages) + extra + 1024);
    return n > 2 ? 2 : (n < 1 ? 1 : n);
  }
  // Upper bound over EVERY call with at most B requests of at most max_ctx tokens (a smaller batch may get more splits per
  // request, so the need is not monotone in B).  Mirrors plan_flat: one wave of blocks, or four, which can only switch on
  // as the context grows; never more splits of a request than a DEC_WARPS-th of its pages.
  static size_t ws_bytes(int sm_count, int max_smem, int B, int n_kv, int max_ctx) {
    const long long slots = (long long)sm_count * ticket_per_sm(2, max_smem, 0), max_tiles = (max_ctx + PAGE - 1) / PAGE;
    size_t best = 0;
    for (int b = 1; b <= B; ++b) {
      const long long units = (long long)b * n_kv;
      long long records = HD == 64 ? 4ll * sm_count : slots;
      if (units * max_tiles >= slots * 4 * 64) records = (4 * slots + units - 1) / units * units;
      const long long most = units * ((max_tiles + DEC_WARPS - 1) / DEC_WARPS);
      if (records > most) records = most;
      if (records < units) records = units;
      const size_t need = ws_need(sm_count, records > units, records);
      if (need > best) best = need;
    }
    return best;
  }
  // Can `need` clusters of `cs` blocks be resident at once?  Asked once per (shape, warps, ring depth, cluster size): the depth
  // decides the shared memory of a block, and an answer for another depth would make a plan depend on earlier calls.
  // The cluster kernel's shared-memory limit is only ever raised: the two ring layouts of one shape (two blocks
  // per SM / one block per SM) need different amounts, and lowering the attribute for the smaller one would
  // make a later launch of the larger one fail.
  // (Function attributes and occupancy answers belong to a device: the caches are indexed by its ordinal.)
  using ClusterKernel = void (*)(const DecodeParams);
  // two blocks per SM (8 warps, head_dim 64) unless the plan uses the one-block-per-SM ring layout
  template <int NW>
  static ClusterKernel cluster_kernel(bool deep) {
    if constexpr (NW == 8 && HD == 64) {
      if (!deep) return lr_attend_decode_cluster_kernel<HD, RK, RV, 8, ROPE, 2>;
    }
    return lr_attend_decode_cluster_kernel<HD, RK, RV, NW, ROPE, 1>;
  }
  template <int NW>
  static cudaError_t ensure_cluster_smem(precc_ctx* ctx, int bytes, bool deep) {
    static bool nonportable_dev[kMaxDevices][2] = {{false}};
    std::lock_guard<std::recursive_mutex> lk(lazy_mu());
    ClusterKernel kern = cluster_kernel<NW>(deep);
    cudaError_t e = raise_smem_limit(ctx, kern, bytes);
    bool& np = nonportable_dev[ctx->device % kMaxDevices][deep ? 1 : 0];
    if (e == cudaSuccess && !np) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) np = true;
    }
    return e;
  }
  template <int NW>
  static bool cluster_fits(precc_ctx* ctx, const DecodePlan& pl, int need) {
    static int cache2[kMaxDevices][DEC_MAX_STAGES + 1][DEC_MAX_CLUSTER + 1] = {{{0}}};  // 0 = unknown, else max active clusters + 1
    std::lock_guard<std::recursive_mutex> lk(lazy_mu());
    int* cached = cache2[ctx->device % kMaxDevices][pl.stages];
    if (cached[pl.cluster] == 0) {
      ClusterKernel kern = cluster_kernel<NW>(pl.deep != 0);
      int n = 0;
      if (ensure_cluster_smem<NW>(ctx, pl.smem, pl.deep != 0) != cudaSuccess) {
        cudaGetLastError();
        cached[pl.cluster] = 1;
        return false;
      }
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(pl.cluster, ctx->sm_count / pl.cluster, 1);
      cfg.blockDim = dim3(NW * 32);
      cfg.dynamicSmemBytes = pl.smem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = pl.cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr; cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
      cached[pl.cluster] = n + 1;
    }
    return cached[pl.cluster] - 1 >= need;
  }
  static constexpr int extra = ROPE ? DecodeCfg<HD, RK, RV>::BK_BYTES + 128 : 0;   // the rotary variant's B_k slice, behind the usual layout

  // ---- ticket kernel: one block per (request, kv head) - no merge, no workspace.  Rings as deep as the blocks that
  //      share an SM allow.
  static DecodePlan plan_whole(precc_ctx* ctx, long long units, int max_tiles) {
    using C = DecodeCfg<HD, RK, RV>;
    const int per_sm = (int)((units + ctx->sm_count - 1) / ctx->sm_count);
    DecodePlan pl{};
    pl.stages = 4;
    while (pl.stages > 2 && (per_sm > 4 ? 4 : per_sm) * (C::ticket_smem(pl.stages) + extra + 1024) > ctx->max_smem_optin) --pl.stages;
    pl.smem = C::ticket_smem(pl.stages) + extra;
    pl.chunk_tiles = max_tiles; pl.max_splits = 1;
    return pl;
  }
  // ---- ticket kernel, up to `want` blocks per unit, their chunk planned from the bound on the lengths
  static DecodePlan plan_split(precc_ctx* ctx, int max_tiles, long long want) {
    DecodePlan pl = plan_whole(ctx, 2 * ctx->sm_count, max_tiles);
    if (want < 1) want = 1;
    int chunk = (int)((max_tiles + want - 1) / want);
    if (chunk < DEC_WARPS) chunk = DEC_WARPS;
    if ((max_tiles + chunk - 1) / chunk > DEC_MAX_SPLITS) chunk = (max_tiles + DEC_MAX_SPLITS - 1) / DEC_MAX_SPLITS;
    pl.chunk_tiles = chunk;
    pl.max_splits = (max_tiles + chunk - 1) / chunk;
    return pl;
  }
  // ---- ticket kernel on a flat grid: one wave of two blocks per SM (four at head_dim 64, whose blocks are small), shared
  //      out by the actual lengths.  Rotary keys take two-page rings: they are bound by issue and gain from the finer
  //      interleaving of short rings (64 units of 2000 .. 16000 tokens: 66 against 70 us).  With many units and plenty of
  //      work four waves planned from the bound level unlike lengths out by themselves, at no cost per block (320 units of
  //      5000 .. 6000 tokens, head_dim 64: 92 against 111 us; 256 units of 4096 .. 32768 tokens: 369 against 381 us).
  static DecodePlan plan_flat(precc_ctx* ctx, int B, int n_kv, int max_tiles) {
    using C = DecodeCfg<HD, RK, RV>;
    const long long units = (long long)B * n_kv;
    DecodePlan pl{};
    pl.stages = ROPE || HD == 64 ? 2 : 4;
    while (pl.stages > 2 && 2 * (C::ticket_smem(pl.stages) + extra + 1024) > ctx->max_smem_optin) --pl.stages;
    pl.smem = C::ticket_smem(pl.stages) + extra;
    const int per_sm = ticket_per_sm(pl.stages, ctx->max_smem_optin, extra);
    const long long slots = (long long)ctx->sm_count * per_sm;
    const long long work = units * max_tiles;
    const bool plenty = work >= slots * 4 * 64;
    if (B > DEC_FLAT_MAX_B || (plenty && units > (ROPE ? (HD == 128 ? 100 : 1) : 63)))
      return plan_split(ctx, max_tiles, plenty ? (4 * slots + units - 1) / units : slots / units);
    long long grid = HD == 64 ? 4ll * ctx->sm_count : slots;
    const long long most = units * ((max_tiles + DEC_WARPS - 1) / DEC_WARPS);   // a split has a page for every warp
    if (grid > most) grid = most;
    if (grid < units) grid = units;
    pl.flat = (int)grid;
    pl.max_splits = 1;
    return pl;
  }
  // ---- cluster kernel with `warps` warps per block at `per_sm` blocks per SM and rings of at most `max_stages` pages: the
  //      widest cluster up to `lim` with all clusters of the grid resident at once.  cluster = 0 when there is none.
  static DecodePlan plan_cluster(precc_ctx* ctx, long long units, int max_tiles, int warps, int per_sm, int max_stages, int lim) {
    using C = DecodeCfg<HD, RK, RV>;
    DecodePlan pl{};
    int stages = max_stages < DEC_MAX_STAGES ? max_stages : DEC_MAX_STAGES;
    if (ctx->decode_stage_cap >= 2 && stages > ctx->decode_stage_cap) stages = ctx->decode_stage_cap;
    while (stages > 2 && per_sm * (C::cluster_smem(warps, stages) + extra + 1024) > ctx->max_smem_optin) --stages;
    pl.smem = C::cluster_smem(warps, stages) + extra;
    if (pl.smem > ctx->max_smem_optin || per_sm * (pl.smem + 1024) > ctx->max_smem_optin + (per_sm == 1 ? 1024 : 0)) return DecodePlan{};
    pl.warps = warps; pl.stages = stages; pl.deep = 2 * (pl.smem + 1024) > ctx->max_smem_optin ? 1 : 0;
    int cs = lim < DEC_MAX_CLUSTER ? lim : DEC_MAX_CLUSTER;
    if (cs > max_tiles) cs = max_tiles;
    if (cs * units > (long long)ctx->sm_count * per_sm) cs = (int)((long long)ctx->sm_count * per_sm / units);
    if (ctx->decode_cluster_cap > 1 && cs > ctx->decode_cluster_cap) cs = ctx->decode_cluster_cap;
    for (; cs >= 1; --cs) {
      pl.cluster = cs;
      if (warps == 8 ? cluster_fits<8>(ctx, pl, (int)units) : cluster_fits<4>(ctx, pl, (int)units)) break;
    }
    pl.cluster = cs;
    pl.max_splits = cs;
    // Short contexts are bound by latency: every request's own pages are shared out evenly.  Long ones are bound by
    // bandwidth: with the chunk of the longest request for all, the blocks of short requests that would finish early do
    // not start, and the longest request gets the bandwidth (24 units of 3188 pages at most: 91 -> 87 us; 12 units of
    // 434 pages at most: 10.7 -> 10.1 us the other way round).
    pl.chunk_tiles = cs >= 1 ? (max_tiles + cs - 1) / cs : 0;
    pl.even = ROPE || (HD == 64 ? max_tiles < 1500 : units * max_tiles < 10000);
    return cs >= 1 ? pl : DecodePlan{};
  }
  // The choice among them, from forced plans of some 1600 shapes (1 .. 64 requests of 100 .. 130000 tokens of unlike
  // length, all layer shapes and ranks; alone, and after a projection in a decode step).  The earlier rules - ticket kernel
  // up to 16 pages, clusters sized for the longest request only, a split planned from the bound - were 20 % above the
  // best plan of each shape on the mean, up to 2x for short contexts; these are 5 % above it.  What decides:
  //   few pages       a block per unit needs no merge; clusters help while most SMs would idle
  //   units <= SMs/2  clusters: merge through distributed shared memory, everything resident in one wave
  //   unlike lengths  the flat grid, once there is enough to read that its schedule and merge are small beside it
  // `units` = (request, kv head) pairs, lengths in pages (mt: the longest request's).  Bounds that are plain numbers of units
  // are those of the 148 SMs that they were measured on.
  static DecodePlan choose(precc_ctx* ctx, int B, int n_kv, int max_ctx) {
    const int sm = ctx->sm_count, mt = (max_ctx + PAGE - 1) / PAGE;
    const long long units = (long long)B * n_kv, work = units * mt;
    auto whole = [&]() { return plan_whole(ctx, units, mt); };
    auto flat = [&]() { return plan_flat(ctx, B, n_kv, mt); };
    auto cluster = [&](int warps, int per_sm, int stages, int lim) { return plan_cluster(ctx, units, mt, warps, per_sm, stages, lim); };
    if (ctx->force_ticket_decode) return flat();
    if (units > sm) {
      // the units fill the machine by themselves; splitting them only evens out unlike lengths
      const int one = ROPE ? (units > 2 * sm ? 64 : 40) : units * 10 > sm * 14 ? (HD == 64 ? 300 : 200) : RK + RV >= 96 ? 200 : HD == 64 ? 64 : 100;
      return mt <= one ? whole() : flat();
    }
    // Few pages: more blocks per unit than it has pages for their warps still pay for small grids (the merge is spread over
    // the cluster, and each block owns fewer output columns), but not beyond about half of the SMs: wide clusters
    // also wait longer for the kernel ahead to leave the SMs.
    const int room = (int)(sm / units), few = room < mt / DEC_WARPS ? room : mt / DEC_WARPS;
    int lim = DEC_MAX_CLUSTER;
    if (ROPE && mt <= 150) lim = mt / 4 < room || room < 2 ? (mt / 4 > 4 ? mt / 4 : 4) : room;
    else if (mt <= 80) lim = 80 / units > 2 ? (int)(80 / units) : 2;
    else if (HD == 64) lim = mt / 12 > 8 ? mt / 12 : 8;
    if (mt <= 80 && lim < few) lim = few;
    DecodePlan pl{};
    if (!ctx->deep_clusters || ctx->deep_always) {       // layout switches of the environment
      if (ctx->deep_always) pl = cluster(8, 1, 4, lim);
      else pl = HD == 64 ? cluster(8, 2, 2, lim) : cluster(4, 2, 3, lim);
      return pl.cluster ? pl : flat();
    }
    if (ROPE) {
      // bound by what the SMs take in from L2: four warps twice per SM reach as many SMs as eight once, in finer pieces; from some work on the flat
      // grid's even shares win
      // (one block each: above three fifths of the SMs that is a fair share of the machine, so it pays up to more pages)
      if (units * 2 > sm && mt <= (units * 5 > 3 * sm ? 48 : 16)) return whole();
      if (units >= 48 && mt <= 12) return whole();
      if (work >= (units >= 56 || RK + RV >= 96 ? 12000 : HD == 64 ? 16000 : 18000)) return flat();
      if (units >= 8 && !(HD == 64 && RK + RV >= 96)) pl = cluster(4, 2, HD == 64 ? 3 : 2, lim);
      if (!pl.cluster) pl = cluster(8, 1, 2, lim);
      return pl.cluster ? pl : flat();
    }
    if (HD == 64) {
      // eight warps twice per SM
      if (units >= 56 && mt <= 16) return whole();
      if (units > 80 && mt > 400) return flat();
      const int wide = RV >= 32 ? (room > 8 ? room : 8) : 12;
      pl = cluster(8, 2, 2, units > 9 && lim > wide ? wide : lim);
      if (!pl.cluster) pl = cluster(8, 1, 3, lim);       // rank 64
      return pl.cluster ? pl : flat();
    }
    if ((units >= 60 && mt <= 20) || (units >= 45 && mt <= 12)) return whole();
    if (units >= 48 && work >= 60000) return flat();
    if (units * 2 > sm) {
      // too many units for two eight-warp blocks each: three four-warp blocks each, two per SM, while that fits
      if (units * 3 <= 2 * sm && mt > 60) {
        pl = cluster(4, 2, 3, 3);
        if (pl.cluster == 3) return pl;
      }
      if (mt <= (RK + RV >= 96 ? 48 : 96)) return whole();
      if (mt > 400) return flat();
      if (RK + RV < 96 && units * 4 <= 3 * sm) return plan_split(ctx, mt, 2 * sm / units);
      pl = cluster(8, 1, 3, 1);
      return pl.cluster ? pl : flat();
    }
    // Eight warps, one block per SM: two or three pages in flight per warp cover the memory's latency.  Clusters of whole SMs
    // do not always use them up (a cluster lives in one GPC: from 45 units on only two blocks each fit, 96 SMs); then two
    // four-warp blocks per SM may reach more of the machine.  They take over where they have three times the blocks, or
    // where the others leave more than a third of the SMs idle and they reach an eighth more (48 units of 320 .. 1000
    // pages: 5 .. 16 % faster than the flat grid; where less is idle the flat grid wins: 56 units of 320 pages 22.6 against
    // 28.1 us, 36 units of 700 pages 35.0 against 42.6).  From some work on the flat grid evens the SMs out by itself
    // wherever clusters use less than ten thirteenths of them.
    pl = cluster(8, 1, work >= 50000 ? 2 : 3, lim);
    const long long reach = pl.cluster * units;          // SMs that have a block
    if (mt >= 100) {
      const DecodePlan p4 = cluster(4, 2, 3, lim);
      if (p4.cluster >= pl.cluster * 3 || (units >= 24 && mt >= 300 && reach * 3 < 2 * sm && p4.cluster * 8 >= pl.cluster * 18)) return p4.cluster ? p4 : flat();
    }
    if (units >= 24 && work >= 30000 && reach * 13 < 10 * sm) return flat();
    return pl.cluster ? pl : flat();
  }
  static int32_t run(precc_ctx* ctx, const DecodeArgs& a) {
    const precc_layer_desc* d = a.d;
    const DecodePlan pl = choose(ctx, a.B, d->n_kv_heads, a.max_ctx);
    // (a plan with one block per unit, and a cluster, use no workspace; the former and the shortest contexts still ask for
    // the one record per unit that the caller's sizing provides at least, so that a missing workspace shows up early)
    const long long units = (long long)a.B * d->n_kv_heads, records = pl.cluster ? units : pl.flat ? pl.flat : units * pl.max_splits;
    const bool split = records > units;                  // pairs of more than one block, which meet at the counters
    if (!pl.cluster || (a.max_ctx + PAGE - 1) / PAGE <= 16) {
      const size_t need = ws_need(ctx->sm_count, split, records);
      if (!a.ws || a.ws_bytes < need) return fail(ctx, PRECC_ERR_WORKSPACE, "decode workspace: need %zu bytes, got %zu", need, a.ws_bytes);
    }
    DecodeParams p;
    p.q = (const __nv_bfloat16*)a.q; p.out = (__nv_bfloat16*)a.out;
    p.agent_id = a.agent_id; p.ctx_len = a.ctx_len; p.block_table = a.block_table; p.first_block = a.first_block;
    p.k_base = (const __nv_bfloat16*)a.cache->k_base; p.v_base = (const __nv_bfloat16*)a.cache->v_base;
    p.lr_k = (const __nv_bfloat16*)a.cache->lr_k; p.lr_v = (const __nv_bfloat16*)a.cache->lr_v;
    p.B_k = (const __nv_bfloat16*)a.B_k; p.B_v = (const __nv_bfloat16*)a.B_v;
    p.tickets = (int32_t*)a.ws;
    p.part = a.ws ? (float*)((char*)a.ws + counter_bytes(ctx->sm_count)) : nullptr;
    p.raw = a.raw;
    p.status = ctx->status;
    p.B = a.B; p.even = pl.even && pl.cluster > 1 ? (unsigned)((1ull << 32) / pl.cluster + 1) : 0u;
    const bool flat = !pl.cluster && pl.flat;
    const size_t n_blocks = flat ? (size_t)pl.flat : (size_t)pl.max_splits * units;
    p.trace = (ctx->trace && n_blocks <= ctx->trace_blocks) ? ctx->trace : nullptr;
    p.n_blocks = a.cache->n_blocks; p.table_stride = a.table_stride;
    p.n_q = d->n_q_heads; p.n_kv = d->n_kv_heads; p.group = d->n_q_heads / d->n_kv_heads; p.n_agents = d->n_agents;
    p.chunk_tiles = pl.chunk_tiles; p.max_splits = pl.max_splits; p.stages = pl.stages; p.max_ctx = a.max_ctx;
    p.pre_stages = (ctx->decode_pre_stages >= 1 && ctx->decode_pre_stages < pl.stages) ? ctx->decode_pre_stages : pl.stages;
    p.scale_log2 = softmax_scale_log2(d); p.s_k = d->lora_scale_k; p.s_v = d->lora_scale_v;
    p.rope = reinterpret_cast<const float4*>(a.rope); p.max_pos = a.max_pos;
    p.bk_off = ROPE ? ((pl.smem - extra + 127) / 128) * 128 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = flat ? dim3(pl.flat) : dim3(pl.max_splits, d->n_kv_heads, a.B);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (pl.cluster) {
      cfg.blockDim = dim3(pl.warps * 32);
      attr[1].id = cudaLaunchAttributeClusterDimension;
      attr[1].val.clusterDim.x = pl.cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
      cfg.numAttrs = 2;
      if (ctx->decode_cluster_policy) {
        // where the blocks of a cluster go inside their GPC: spread over as many SMs as possible, or packed
        attr[2].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
        attr[2].val.clusterSchedulingPolicyPreference =
            ctx->decode_cluster_policy == 1 ? cudaClusterSchedulingPolicySpread : cudaClusterSchedulingPolicyLoadBalancing;
        cfg.numAttrs = 3;
      }
      if (pl.warps == 8) {
        PRECC_CUDA(ctx, ensure_cluster_smem<8>(ctx, pl.smem, pl.deep != 0));
        PRECC_CUDA(ctx, cudaLaunchKernelEx(&cfg, cluster_kernel<8>(pl.deep != 0), p));
      } else {
        PRECC_CUDA(ctx, ensure_cluster_smem<4>(ctx, pl.smem, pl.deep != 0));
        PRECC_CUDA(ctx, cudaLaunchKernelEx(&cfg, cluster_kernel<4>(pl.deep != 0), p));
      }
    } else {
      auto kern = flat ? lr_attend_decode_kernel<HD, RK, RV, ROPE, true> : lr_attend_decode_kernel<HD, RK, RV, ROPE, false>;
      cfg.blockDim = dim3(DEC_WARPS * 32);
      PRECC_CUDA(ctx, raise_smem_limit(ctx, kern, pl.smem));
      if (a.clear_counters && split) PRECC_CUDA(ctx, cudaMemsetAsync(p.tickets, 0, counter_bytes(ctx->sm_count), a.stream));
      PRECC_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, p));
    }
    return PRECC_OK;
  }
};

template <int HD, int RK, int RV>
struct DecodeRun : DecodeRunT<HD, RK, RV, false> {};
// Rotary keys: without a key-side adapter (or for the adapter-free view) the rotated base cache is all
// there is, and the position-free kernel is already exact.
template <int HD, int RK, int RV>
struct DecodeRunRope {
  static int32_t run(precc_ctx* ctx, const DecodeArgs& a) {
    if constexpr (RK > 0) return DecodeRunT<HD, RK, RV, true>::run(ctx, a);
    else return DecodeRunT<HD, RK, RV, false>::run(ctx, a);
  }
};


template <int HD, int RK, int RV>
struct DecodeWs {
  static int32_t run(precc_ctx*, const WsQuery& w) {
    *w.out = DecodeRun<HD, RK, RV>::ws_bytes(w.sm_count, w.max_smem, w.B, w.n_kv, w.max_ctx);
    return PRECC_OK;
  }
};

}  // namespace precc

#define PRECC_DEFINE_DECODE_UNIT(HD)                                                                          \
  namespace precc {                                                                                           \
  int32_t decode_run_hd##HD(precc_ctx* ctx, const DecodeArgs& a) {                                            \
    if (a.rope) return dispatch_ranks<DecodeRunRope, HD>(ctx, a.d->rank_k, a.d->rank_v, a);                   \
    return dispatch_ranks<DecodeRun, HD>(ctx, a.d->rank_k, a.d->rank_v, a);                                   \
  }                                                                                                           \
  int32_t decode_ws_hd##HD(precc_ctx* ctx, int rk, int rv, const WsQuery& w) {                                \
    return dispatch_ranks<DecodeWs, HD>(ctx, rk, rv, w);                                                      \
  }                                                                                                           \
  }
