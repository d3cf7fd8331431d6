"""The work that users of this library have it do, as cases that can be timed and compared.

Four kinds of pass, all through ``paper_2609_34054_b200.binding``:

* ``decode``      one attention call of a decode step: a batch of requests over base cache + own LR cache
* ``step``        one decode step of a stack of layers: per layer the new tokens' projection and the attention
* ``turn``        one layer of a turn's prefill: projection of the S new tokens, their attention over T cached
                  tokens, and (``rebase``) the re-projection of the adapter-free hidden states
* ``precompute``  the LR rows of every agent for a processed segment

Layer shapes are those of the repository's workloads (d_model 1024 / 2048 / 3584 / 4096), sizes those of its
benchmark, sweep and trace replay.  Everything is drawn on the device from the seed; lengths come from the case alone,
so that the work of a case does not depend on the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2609_34054_b200 import inputs as I
from paper_2609_34054_b200.binding import Cache, Precc, layer_desc

PAGE = I.PAGE

# (d_model, query heads, kv heads, head_dim) of the repository's layers
SMALL, ONE_B, SEVEN_B, EIGHT_B = (1024, 8, 2, 128), (2048, 32, 8, 64), (3584, 28, 4, 128), (4096, 32, 8, 128)


def _case(kind, shape, agents, rank_k, rank_v, **sizes):
    d, n_q, n_kv, hd = shape
    return dict(kind=kind, d_model=d, n_q=n_q, n_kv=n_kv, head_dim=hd, agents=agents, rank_k=rank_k, rank_v=rank_v, **sizes)


def _decode(shape, agents, rank_k, rank_v, batch, ctx_min, ctx_max, paged, rope):
    return _case("decode", shape, agents, rank_k, rank_v, batch=batch, ctx_min=ctx_min, ctx_max=ctx_max, paged=paged, rope=rope)


def _step(shape, agents, rank_k, rank_v, layers, batch, ctx_min, ctx_max, double, rope, graph):
    return _case("step", shape, agents, rank_k, rank_v, layers=layers, batch=batch, ctx_min=ctx_min, ctx_max=ctx_max,
                 double=double, rope=rope, graph=graph)


def _turn(shape, agents, rank_k, rank_v, new, ctx, paged, rope, workspace, rebase):
    return _case("turn", shape, agents, rank_k, rank_v, new=new, ctx=ctx, paged=paged, rope=rope, workspace=workspace, rebase=rebase)


def _precompute(shape, agents, rank_k, rank_v, rows):
    return _case("precompute", shape, agents, rank_k, rank_v, rows=rows)


def listed():
    return [
        # one decode query per agent over a short shared context: the smallest call there is
        dict(_decode(SMALL, 3, 8, 8, 3, 256, 256, False, False), name="decode-tiny"),
        # a handful of requests of unlike length, LoRA on the query and value projections only (the paper's default)
        dict(_decode(EIGHT_B, 3, 0, 8, 7, 700, 3100, True, False), name="decode-few-ragged"),
        # concurrent serving: 64 requests of 4k..32k tokens, agents mixed, paged caches
        dict(_decode(SEVEN_B, 8, 16, 16, 64, 4096, 32768, True, False), name="decode-serving"),
        # rotary keys, a small batch of medium contexts
        dict(_decode(EIGHT_B, 4, 16, 16, 8, 2000, 16000, True, True), name="decode-rotary"),
        # single-stream generation: a 16-layer step replayed as a CUDA graph, as the benchmark and the trace replay do
        dict(_step(ONE_B, 4, 16, 16, 16, 1, 8192, 8192, False, False, True), name="step-single-graph"),
        # double batching (the turn's adapted and adapter-free sequences in one batch), called layer by layer
        dict(_step(EIGHT_B, 4, 32, 32, 8, 1, 5000, 5000, True, False, False), name="step-double"),
        # a tool observation or plan / reflect input: few new tokens over a long shared context
        dict(_turn(EIGHT_B, 4, 32, 32, 64, 16384, False, False, False, False), name="turn-short"),
        # an ordinary turn: 512 new tokens over 32k, then the base rows rebuilt from adapter-free hidden states
        dict(_turn(EIGHT_B, 4, 32, 32, 512, 32768, False, False, False, True), name="turn-rebase"),
        # a turn of odd length over a paged context with a caller workspace, head_dim 64
        dict(_turn(ONE_B, 4, 16, 16, 301, 5003, True, False, True, False), name="turn-odd"),
        # rotary keys through the key scratch, seven query heads per kv head
        dict(_turn(SEVEN_B, 8, 16, 16, 200, 8000, True, True, False, False), name="turn-rotary"),
        # retrieved context handed to an agent: a long segment over what is already there
        dict(_turn(EIGHT_B, 3, 32, 32, 8192, 24576, False, False, False, False), name="turn-long"),
        # LR rows of all agents for a whole shared context
        dict(_precompute(EIGHT_B, 4, 32, 32, 32768), name="precompute-context"),
    ]


_DECODE_BYTES = 2.5e9      # caches of a drawn decode or step: about those of the serving batch
_TURN_FLOPS = 4.9e12       # a drawn turn: about the long turn


def _log_int(rng, low, high):
    return max(low, min(high, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    kind = rng.choices(("decode", "step", "turn", "precompute"), (4, 2, 5, 1))[0]
    shape = rng.choice((SMALL, ONE_B, SEVEN_B, EIGHT_B, EIGHT_B))
    agents, rank_v = rng.choice((2, 3, 4, 8, 16)), rng.choice((8, 16, 32, 64))
    rank_k = rank_v if kind == "precompute" or rng.random() < 0.75 else 0
    rope = rank_k > 0 and rng.random() < 0.25
    while True:
        if kind == "decode":
            ctx_max = _log_int(rng, 256, 131072)
            c = _decode(shape, agents, rank_k, rank_v, _log_int(rng, 1, 64), max(1, int(ctx_max * rng.uniform(0.1, 1.0))), ctx_max,
                        rng.random() < 0.67, rope)
            fits = work(c)["bytes"] <= _DECODE_BYTES
        elif kind == "step":
            ctx_max, double = _log_int(rng, 256, 32768), rng.random() < 0.33
            c = _step(shape, agents, rank_k, rank_v, _log_int(rng, 2, 16), _log_int(rng, 1, 16), max(1, int(ctx_max * rng.uniform(0.1, 1.0))),
                      ctx_max, double, rope and not double, rng.random() < 0.5)
            fits = work(c)["bytes"] <= _DECODE_BYTES
        elif kind == "turn":
            c = _turn(shape, agents, rank_k, rank_v, _log_int(rng, 16, 8192), 0 if rng.random() < 0.1 else _log_int(rng, 256, 65536),
                      rng.random() < 0.5, rope, not rope and rng.random() < 0.33, not rope and rng.random() < 0.25)
            fits = work(c)["flops"] <= _TURN_FLOPS
        else:
            c, fits = _precompute(shape, agents, rank_k, rank_v, _log_int(rng, 128, 32768)), True
        if fits:
            return c


def _geometry(c):
    return I.Geometry(d_model=c["d_model"], n_q=c["n_q"], n_kv=c["n_kv"], hd=c["head_dim"], n_agents=c["agents"],
                      rank_k=c["rank_k"], rank_v=c["rank_v"], alpha=2.0 * max(c["rank_k"], c["rank_v"]))


def _contexts(c):
    """Lengths spread over [ctx_min, ctx_max] in an unordered but fixed way."""
    span = c["ctx_max"] - c["ctx_min"]
    return [c["ctx_max"] - int(span * ((b * 0.6180339887498949) % 1.0)) for b in range(c["batch"])]


def _pages(n):
    return (n + PAGE - 1) // PAGE


# ------------------------------------------------------------------------------------------------- inputs
_context = None


def _px():
    """A program has one library context per device."""
    global _context
    if _context is None:
        _context = Precc(0)
    return _context


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1_000_003 + 12_345)
    return g


def _normal(gen, shape, std=1.0):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)


def _weights(gen, geo):
    d, w, n = geo.d_model, geo.kv_width, geo.n_agents
    return dict(W_k=_normal(gen, (d, w), 0.02), W_v=_normal(gen, (d, w), 0.02),
                A_k=_normal(gen, (n, d, geo.rank_k), d ** -0.5) if geo.rank_k else None, A_v=_normal(gen, (n, d, geo.rank_v), d ** -0.5),
                B_k=_normal(gen, (n, geo.rank_k, w), 0.02) if geo.rank_k else None, B_v=_normal(gen, (n, geo.rank_v, w), 0.02))


def _pools(gen, geo, layers, n_blocks):
    """Cache contents of `layers` layers, distributed as H.W and H.A are; [layers, ...] each."""
    sig = 0.02 * geo.d_model ** 0.5
    pool = dict(k=_normal(gen, (layers, n_blocks, geo.n_kv, PAGE, geo.hd), sig), v=_normal(gen, (layers, n_blocks, geo.n_kv, PAGE, geo.hd), sig),
                lr_k=_normal(gen, (layers, geo.n_agents, n_blocks, PAGE, geo.rank_k)) if geo.rank_k else None,
                lr_v=_normal(gen, (layers, geo.n_agents, n_blocks, PAGE, geo.rank_v)))
    caches = [Cache.from_tensors(geo, pool["k"][l], pool["v"][l], None if pool["lr_k"] is None else pool["lr_k"][l], pool["lr_v"][l])
              for l in range(layers)]
    return pool, caches


def _written(pool, first):
    """The cache blocks from physical block `first` on: those that a pass writes to."""
    return [pool["k"][:, first:], pool["v"][:, first:], None if pool["lr_k"] is None else pool["lr_k"][:, :, first:], pool["lr_v"][:, :, first:]]


def _i32(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _table(pages, perm):
    """Block tables of requests that own pages[b] blocks each, handed out from `perm`; unused entries -1."""
    table = torch.full((len(pages), max(pages)), -1, dtype=torch.int32)
    at = 0
    for b, n in enumerate(pages):
        table[b, :n] = perm[at:at + n]
        at += n
    return table


def _prepare_decode(c, seed):
    px, geo, gen = _px(), _geometry(c), _generator(seed)
    ctx, host = _contexts(c), torch.Generator().manual_seed(seed)
    pages = [_pages(t) for t in ctx]
    _, caches = _pools(gen, geo, 1, sum(pages))
    w = _weights(gen, geo)
    desc, table, first = layer_desc(geo), None, None
    if c["paged"]:
        table = _table(pages, torch.randperm(sum(pages), generator=host).to(torch.int32)).cuda()
    else:
        first = _i32([sum(pages[:b]) for b in range(len(pages))])
    q = _normal(gen, (c["batch"], geo.n_q, geo.hd))
    agent = torch.randint(0, geo.n_agents, (c["batch"],), generator=host, dtype=torch.int32).cuda()
    args = (desc, q, agent, _i32(ctx), max(ctx), w["B_k"], w["B_v"])
    rope = (I.rope_table(max(ctx), geo.hd),) if c["rope"] else ()
    out, ws = torch.empty_like(q), px.decode_workspace(desc, c["batch"], max(ctx))
    call = px.lr_attend_decode_rope if c["rope"] else px.lr_attend_decode
    return dict(call=call, args=args + rope + (caches[0], out, ws, table, first), out=out)


def _run_decode(s):
    s["call"](*s["args"])
    return s["out"]


def _prepare_step(c, seed):
    px, geo, gen = _px(), _geometry(c), _generator(seed)
    ctx, host, B, L = _contexts(c), torch.Generator().manual_seed(seed), c["batch"], c["layers"]
    # physical blocks: the requests' full pages in random order, then the page each request is writing to; with double
    # batching also the private page of each adapted sequence
    full = [_pages(t) - 1 for t in ctx]
    n_full = sum(full)
    n_blocks = n_full + B * (2 if c["double"] else 1)
    table = torch.full((B, max(full) + 1), -1, dtype=torch.int32)
    perm = torch.randperm(n_full, generator=host).to(torch.int32)
    for b, n in enumerate(full):
        at = sum(full[:b])
        table[b, :n] = perm[at:at + n]
        table[b, n] = n_full + b
    agent = torch.randint(0, geo.n_agents, (B,), generator=host, dtype=torch.int32)
    slots = torch.tensor([(n_full + b) * PAGE + (t - 1) % PAGE for b, t in enumerate(ctx)], dtype=torch.int32)
    rows, masks, copies = B, None, None
    if c["double"]:
        private = table.clone()
        for b, n in enumerate(full):
            private[b, n] = n_full + B + b
        table, rows = torch.cat([private, table]), 2 * B           # the adapted sequences, then the adapter-free ones
        own = torch.ones(B, dtype=torch.int64) << agent.to(torch.int64)
        masks = torch.cat([own, ((1 << geo.n_agents) - 1) & ~own]).cuda()
        copies = torch.cat([slots, torch.full((B,), -1, dtype=torch.int32)]).cuda()
        slots = torch.cat([slots + B * PAGE, slots])
        agent, ctx = torch.cat([agent, torch.full((B,), -1, dtype=torch.int32)]), ctx + ctx
    pool, caches = _pools(gen, geo, L, n_blocks)
    desc = layer_desc(geo)
    H, q = _normal(gen, (L, rows, geo.d_model)), _normal(gen, (L, rows, geo.n_q, geo.hd))
    weights = []
    for _ in range(L):
        w = _weights(gen, geo)
        weights.append((px.pack_turn_weights(geo, w["W_k"], w["W_v"], w["A_k"], w["A_v"]), w["B_k"], w["B_v"]))
    s = dict(px=px, desc=desc, layers=L, H=[H[l] for l in range(L)], q=[q[l] for l in range(L)], weights=weights, caches=caches,
             slots=slots.cuda(), masks=masks, copies=copies, agent=agent.cuda(), ctx=_i32(ctx), max_ctx=max(ctx), table=table.cuda(),
             positions=_i32([t - 1 for t in ctx]), rope=I.rope_table(max(ctx), geo.hd) if c["rope"] else None,
             ws=px.decode_workspace(desc, rows, max(ctx)), graph=None)
    out = torch.empty_like(q)
    s["out"], s["outputs"] = [out[l] for l in range(L)], [out] + _written(pool, n_full)
    if c["graph"]:
        _step_calls(s)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _step_calls(s)
    return s


def _step_calls(s):
    px, desc = s["px"], s["desc"]
    for l in range(s["layers"]):
        WA, B_k, B_v = s["weights"][l]
        cache, out = s["caches"][l], s["out"][l]
        if s["masks"] is not None:
            px.turn_project_rows(desc, s["H"][l], WA, cache, s["slots"], s["masks"], s["copies"])
        elif s["rope"] is not None:
            px.turn_project_rope(desc, s["H"][l], WA, cache, s["rope"], slot_mapping=s["slots"], positions=s["positions"])
        else:
            px.turn_project(desc, s["H"][l], WA, cache, slot_mapping=s["slots"])
        if s["rope"] is not None:
            px.lr_attend_decode_rope(desc, s["q"][l], s["agent"], s["ctx"], s["max_ctx"], B_k, B_v, s["rope"], cache, out, s["ws"], s["table"])
        else:
            px.lr_attend_decode(desc, s["q"][l], s["agent"], s["ctx"], s["max_ctx"], B_k, B_v, cache, out, s["ws"], s["table"])


def _run_step(s):
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        _step_calls(s)
    return s["outputs"]


def _prepare_turn(c, seed):
    px, geo, gen = _px(), _geometry(c), _generator(seed)
    S, T, host = c["new"], c["ctx"], torch.Generator().manual_seed(seed)
    n_blocks, old = _pages(T + S), T // PAGE
    pool, caches = _pools(gen, geo, 1, n_blocks)
    w, desc = _weights(gen, geo), layer_desc(geo)
    # paged: the pages in front of the new tokens, and those the new tokens go to, each in random order
    table = slots = None
    if c["paged"]:
        table = torch.cat([torch.randperm(old, generator=host), old + torch.randperm(n_blocks - old, generator=host)]).to(torch.int32)
        at = torch.arange(T, T + S)
        slots = (table[at // PAGE] * PAGE + (at % PAGE).to(torch.int32)).to(torch.int32).cuda()
        table = table.cuda()
    q = _normal(gen, (S, geo.n_q, geo.hd))
    s = dict(px=px, desc=desc, cache=caches[0], H=_normal(gen, (S, geo.d_model)), H_neutral=None, q=q, out=torch.empty_like(q), T=T,
             agent=int(torch.randint(0, geo.n_agents, (1,), generator=host)), table=table, slots=slots, rope=None, ws=None,
             WA=px.pack_turn_weights(geo, w["W_k"], w["W_v"], w["A_k"], w["A_v"]), B_k=w["B_k"], B_v=w["B_v"])
    if c["rebase"]:
        s["W"], s["H_neutral"] = px.pack_base_weights(geo, w["W_k"], w["W_v"]), _normal(gen, (S, geo.d_model))
    if c["rope"]:
        s["rope"] = I.rope_table(T + S, geo.hd)
        s["scratch"] = torch.empty(px.prefill_rope_scratch_bytes(desc, T, S), dtype=torch.uint8, device="cuda")
    if c["workspace"]:
        s["ws"] = torch.empty(max(256, px.prefill_ws_bytes(desc, S)), dtype=torch.uint8, device="cuda")
    s["outputs"] = [s["out"]] + _written(pool, old)
    return s


def _run_turn(s):
    px, desc, cache, T = s["px"], s["desc"], s["cache"], s["T"]
    if s["rope"] is not None:
        px.turn_project_rope(desc, s["H"], s["WA"], cache, s["rope"], start_slot=T, slot_mapping=s["slots"], start_pos=T)
        px.lr_attend_prefill_rope_scratch(desc, s["q"], s["agent"], T, s["B_k"], s["B_v"], s["rope"], cache, s["out"], s["scratch"], s["table"])
    else:
        px.turn_project(desc, s["H"], s["WA"], cache, start_slot=T, slot_mapping=s["slots"])
        if s["ws"] is not None:
            px.lr_attend_prefill_ws(desc, s["q"], s["agent"], T, s["B_k"], s["B_v"], cache, s["out"], s["ws"], s["table"])
        else:
            px.lr_attend_prefill(desc, s["q"], s["agent"], T, s["B_k"], s["B_v"], cache, s["out"], s["table"])
    if s["H_neutral"] is not None:
        px.rebase_project(desc, s["H_neutral"], s["W"], cache, start_slot=T, slot_mapping=s["slots"])
    return s["outputs"]


def _prepare_precompute(c, seed):
    px, geo, gen = _px(), _geometry(c), _generator(seed)
    w = _weights(gen, geo)
    cache = Cache(geo, _pages(c["rows"]), fill=0.0)
    return dict(px=px, args=(layer_desc(geo), _normal(gen, (c["rows"], geo.d_model)), px.pack_adapters(geo, w["A_k"], w["A_v"]), cache),
                outputs=[cache.lr_k, cache.lr_v])


def _run_precompute(s):
    s["px"].lr_precompute(*s["args"])
    return s["outputs"]


_KINDS = {"decode": (_prepare_decode, _run_decode), "step": (_prepare_step, _run_step), "turn": (_prepare_turn, _run_turn),
          "precompute": (_prepare_precompute, _run_precompute)}


def prepare(case, seed):
    prepare_kind, run_kind = _KINDS[case["kind"]]
    return run_kind, prepare_kind(case, seed)


def run(state):
    run_kind, s = state
    return run_kind(s)


# ------------------------------------------------------------------------------------------- work and accuracy
def work(case):
    """Bytes (bf16 tensors, int32 indices, fp32 rotary table) and flops of one pass."""
    g = _geometry(case)
    lr, base = g.rank_k + g.rank_v, 2 * g.kv_width
    n_out, b_slice = base + g.n_agents * lr, lr * g.kv_width * 2          # fused projection width; one agent's B factors

    def project(rows, columns):
        return 2 * (rows * g.d_model + columns * g.d_model + rows * columns), 2 * rows * g.d_model * columns

    def attend(queries, pairs, stored, agents, table_rows):
        """`pairs` (query, key) pairs per query head, `stored` cached tokens read, rows of the rotary table."""
        byts = stored * (base + lr) * 2 + queries * 2 * g.n_q * g.hd * 2 + agents * b_slice + table_rows * g.hd * 4
        return byts, 4 * g.n_q * (g.hd + lr / 2) * pairs

    if case["kind"] == "precompute":
        parts, times = [project(case["rows"], g.n_agents * lr)], 1
    elif case["kind"] == "turn":
        S, T = case["new"], case["ctx"]
        parts, times = [project(S, n_out), attend(S, S * T + S * (S + 1) / 2, T, 1, T + S if case["rope"] else 0)], 1
        if case["rebase"]:
            parts.append(project(S, base))
    else:
        ctx, B = _contexts(case), case["batch"]
        twice = 2 if case.get("double") else 1                            # the two sequences of a turn share their context
        parts = [attend(B * twice, twice * sum(ctx), sum(ctx), min(B, g.n_agents), max(ctx) if case["rope"] else 0)]
        parts.append((4 * sum(_pages(t) for t in ctx) * twice, 0))
        times = case.get("layers", 1)
        if case["kind"] == "step":
            parts.append(project(B * twice, n_out))
    return {"bytes": times * sum(p[0] for p in parts), "flops": times * sum(p[1] for p in parts)}


def tolerance(case):
    """All tensors are bf16 with fp32 accumulation; softmax weights and folded queries are rounded to bf16 on the way."""
    return {"rel": 1e-2}
