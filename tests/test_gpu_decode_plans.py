"""How decode attention is split over the GPU: the flat grid's schedule and the other plans at their edges, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import lrkv_oracle as O
from paper_2609_34054_b200 import inputs as I
from paper_2609_34054_b200.binding import Cache, Precc, layer_desc

from harness import assert_close, f64

pytestmark = pytest.mark.gpu

TICKET = {"PRECC_DECODE": "ticket"}          # no clusters: the flat grid (up to 256 requests) whatever the sizes


def _ragged(B, low, high):
    return [low + (b * 7919 + 13) % (high - low + 1) for b in range(B)]


_PLANS = [
    # plan taken, env, head_dim, kv heads, query heads per kv head, rank, lengths, requests rejected on the device
    ("flat", TICKET, 64, 1, 4, 16, [1], ()),                                     # one page, one block
    ("flat", TICKET, 128, 2, 4, 16, [127, 129], ()),                             # fewer pages than a block has warps
    ("flat", TICKET, 64, 2, 2, 8, [9000], ()),                                   # one request over the whole grid
    ("flat", TICKET, 128, 3, 2, 32, [700, 16, 4000, 17, 1300], (2,)),            # a rejected request in the middle counts as one page
    ("flat", TICKET, 64, 1, 4, 0, _ragged(32, 1, 900), ()),                      # one request per lane of the schedule
    ("flat", TICKET, 64, 2, 8, 64, _ragged(33, 1, 900), (0, 32)),
    ("flat", TICKET, 64, 1, 2, 16, _ragged(256, 1, 1500), (255,)),               # the most the schedule handles
    ("split", TICKET, 64, 1, 2, 16, _ragged(257, 1, 1500), ()),                  # one more: split from the bound (one block each)
    ("flat", {}, 64, 2, 4, 16, _ragged(80, 300, 1600), ()),                      # more units than SMs, unlike lengths
    ("split", {}, 64, 2, 4, 16, _ragged(40, 60, 250), ()),                       # one block per unit
    ("split 2", {}, 128, 2, 4, 16, _ragged(50, 700, 1700), ()),                  # two blocks per unit, planned from the bound
    ("cluster 1", {}, 128, 2, 4, 64, _ragged(50, 700, 1700), ()),                # one cluster block per unit
    ("cluster", {}, 128, 8, 4, 16, [10500, 900], ()),                            # clusters, the longest request's chunk for all
    ("cluster", {}, 128, 2, 4, 16, [256, 30, 250], ()),                          # clusters, every request shared out evenly
    # where whole-SM clusters leave SMs idle: three blocks per unit, then five smaller ones while a third is idle, then the flat grid
    ("cluster", {}, 128, 4, 4, 16, _ragged(11, 5600, 12000), ()),
    ("cluster", {}, 128, 4, 4, 16, _ragged(12, 5600, 12000), ()),
    ("flat", {}, 128, 4, 4, 16, _ragged(13, 5600, 12000), ()),
]


def _plan_taken(px, trace, units, hd, pages):
    """From the stamps of the last call: how many blocks it started, and whether they were clusters (only those write entry 15)."""
    t = trace.cpu()
    blocks, cluster = int((t[:, 0] != 0).sum()), bool((t[:, 15] != 0).any())
    each = blocks // units
    if cluster:
        assert blocks == each * units
        return {"cluster", f"cluster {each}"}
    slots = (4 if hd == 64 else 2) * px.sm_count
    flat = {"flat"} if blocks == max(units, min(slots, units * ((pages + 3) // 4))) else set()
    return flat | ({"split" if each == 1 else f"split {each}"} if blocks == each * units else set())


@pytest.mark.parametrize("plan,env,hd,n_kv,G,r,ctx,rejected", _PLANS, ids=[str(i) for i in range(len(_PLANS))])
def test_every_plan_against_the_oracle(monkeypatch, plan, env, hd, n_kv, G, r, ctx, rejected):
    """Paged caches (pages shared between requests, in mixed order).  The tolerance is that of every other decode test:
    bf16 inputs and softmax weights, fp32 accumulation."""
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    px = Precc(0)                                        # the switch is read when a context is created
    try:
        geo = I.Geometry(512, G * n_kv, n_kv, hd, 2, r, r, alpha=2.0 * max(r, 1))
        B, T = len(ctx), max(ctx)
        pages = (T + 15) // 16
        c = I.direct_caches(pages + 5, geo, 83, f"plan.{hd}.{n_kv}.{r}")
        cache = Cache.from_tensors(geo, c["k_base"].cuda(), c["v_base"].cuda(), c["lr_k"].cuda() if r else None,
                                   c["lr_v"].cuda() if r else None)
        w, desc = I.layer_weights(geo, 83, "plan"), layer_desc(geo)
        B_k, B_v = (w["B_k"].cuda(), w["B_v"].cuda()) if r else (None, None)
        q = I.queries(B, geo, 83, "plan.q", gain=4.0)
        table = torch.stack([torch.roll(torch.arange(pages + 5), b)[:pages] for b in range(B)]).to(torch.int32)
        lengths = torch.tensor([8 * T if b in rejected else n for b, n in enumerate(ctx)], dtype=torch.int32).cuda()
        agent = torch.tensor([b % 2 for b in range(B)], dtype=torch.int32).cuda()
        ws = px.decode_workspace(desc, B, T)
        out, again = torch.full_like(q, float("nan"), device="cuda"), torch.full_like(q, float("nan"), device="cuda")
        trace = torch.zeros(4096, 16, dtype=torch.int64, device="cuda")
        for o in (out, again):
            px.lr_attend_decode(desc, q.cuda(), agent, lengths, T, B_k, B_v, cache, o, ws, table.cuda())
            px.set_trace_buffer(trace)
        px.set_trace_buffer(None)
        assert plan in _plan_taken(px, trace, B * n_kv, hd, pages)
        assert px.poll_status() == (1 if rejected else 0)
        assert torch.equal(out, again)
        check = {b for b in (0, 1, B // 2, B - 2, B - 1, int(np.argmax(ctx)), int(np.argmin(ctx))) if 0 <= b < B}
        for b in sorted(check | set(rejected)):
            if b in rejected:
                assert (out[b] == 0).all()
                continue
            own, n, a = table[b].long(), ctx[b], b % 2
            for g in {0, n_kv - 1}:
                cols, zero = slice(g * hd, (g + 1) * hd), np.zeros((1, hd))
                rows = lambda x: f64(x.reshape(-1, x.shape[-1]))[:n]
                lr = lambda x: rows(x[a][own]) if r else np.zeros((n, 1))
                ref = O.attend_from_caches(f64(q[b, g * G:(g + 1) * G]), rows(c["k_base"][own, g]), rows(c["v_base"][own, g]),
                                           lr(c["lr_k"]), lr(c["lr_v"]), f64(w["B_k"][a][:, cols]) if r else zero,
                                           f64(w["B_v"][a][:, cols]) if r else zero, geo.scale_k if r else 0.0,
                                           geo.scale_v if r else 0.0, 1)
                assert_close(f64(out)[b, g * G:(g + 1) * G], ref, f"request {b} of {n} tokens, head {g}")
    finally:
        px.close()


@pytest.mark.parametrize("hd,r,rope,env", [(128, 16, False, TICKET), (64, 8, False, TICKET), (64, 64, False, TICKET), (128, 16, True, {})])
def test_one_workspace_for_growing_batches_and_other_layers(monkeypatch, hd, r, rope, env):
    """Split decode calls of 8 .. 256 (request, kv head) pairs, of two layer shapes, on one workspace: what a call leaves in it
    (records) must not reach what a later call expects to be zero (arrival counters).  A first pass on a workspace
    of its own is the reference, itself checked against the oracle."""
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    px = Precc(0)
    try:
        runs, need, T = [], 0, 4000
        for n_kv in (8, 2):
            geo = I.Geometry(512, 2 * n_kv, n_kv, hd, 2, r, r, alpha=2.0 * r)
            desc, pages, w = layer_desc(geo), T // 16, I.layer_weights(geo, 84, "ws")
            c = I.direct_caches(pages + 5, geo, 84, f"ws.{hd}.{n_kv}.{r}")
            cache = Cache.from_tensors(geo, *(c[k].cuda() for k in ("k_base", "v_base", "lr_k", "lr_v")))
            for B in (1, 8, 16, 32):
                ctx = [T] + _ragged(B - 1, 1500, T)
                table = torch.stack([torch.roll(torch.arange(pages + 5), b)[:pages] for b in range(B)]).to(torch.int32)
                q = I.queries(B, geo, 84, "ws.q", gain=4.0)
                args = [desc, q.cuda(), torch.tensor([b % 2 for b in range(B)], dtype=torch.int32).cuda(),
                        torch.tensor(ctx, dtype=torch.int32).cuda(), T, w["B_k"].cuda(), w["B_v"].cuda()]
                runs.append((args + ([I.rope_table(T, hd)] if rope else []) + [cache], table.cuda(), B))
                need = max(need, px.decode_workspace(desc, 32, T).numel())
                if not rope and B in (1, 32):
                    own = px.decode_workspace(desc, B, T)
                    out = torch.full_like(args[1], float("nan"))
                    px.lr_attend_decode(*args, cache, out, own, table.cuda())
                    b, g = B - 1, n_kv - 1
                    pg, n, a, cols = table[b].long(), ctx[b], b % 2, slice(g * hd, (g + 1) * hd)
                    rows = lambda x: f64(x.reshape(-1, x.shape[-1]))[:n]
                    ref = O.attend_from_caches(f64(q[b, 2 * g:2 * g + 2]), rows(c["k_base"][pg, g]), rows(c["v_base"][pg, g]),
                                               rows(c["lr_k"][a][pg]), rows(c["lr_v"][a][pg]), f64(w["B_k"][a][:, cols]),
                                               f64(w["B_v"][a][:, cols]), geo.scale_k, geo.scale_v, 1)
                    assert_close(f64(out)[b, 2 * g:2 * g + 2], ref, f"batch of {B}, {n} tokens")
        shared = torch.zeros(need, dtype=torch.uint8, device="cuda")
        call = px.lr_attend_decode_rope if rope else px.lr_attend_decode
        for _ in range(2):
            for args, table, B in runs:
                own = px.decode_workspace(args[0], B, T)
                want, out = (torch.full_like(args[1], float("nan")) for _ in range(2))
                call(*args, want, own, table)
                call(*args, out, shared, table)
                assert not torch.isnan(out).any() and torch.equal(out, want), f"batch of {B}, {args[0].n_kv_heads} kv heads"
        assert px.poll_status() == 0
    finally:
        px.close()
