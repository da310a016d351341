"""What the library is timed on: the calls a user of the eviction path makes, from the smallest to the largest.

A user's program is a decode loop over the layers of a model.  Every step of it calls ``skipkv_decode_step`` once per
layer (or ``skipkv_append`` and ``skipkv_decode_attn``; over a paged cache the ``_paged`` forms) and, where a token closes
a sentence, ``skipkv_table_step``.  When the cache has outgrown its budget -- after a long prompt, then every 128 steps or
so -- it scores every layer, selects the sentences to keep and compacts the cache in place.  The sizes are those of
``workloads.config``: 1 (one sequence, 2048 tokens), 2 and 3 (ten sequences of 16K to 32K tokens, budget 4096), 4 (the
decode loop around budget 2048) and 5 (sixteen sequences of 32K to 64K tokens, five query heads per KV head, window 64,
budget 8192).

Keys of a case:
  op      step | attn | score | evict | token_red | table
  cache   slab (contiguous) | paged (128-row pages) | static (attn without a workspace)
  batch, hq, hk, window, d_model, layers
  lo, hi  cached tokens per sequence, evenly spread over the sequences between the two
  budget, fill (exactly-B selection), lam (score: penalty from the pooled keys or from the lookup table)
  sents   sentence lengths: "uniform" 8..96, or "geometric" 4 + Geom(20) up to 128; dup: share of near-duplicates

The sequences' lengths depend on the case alone; everything else is drawn from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_07993_b200 import binding as B
from paper_2512_07993_b200 import workloads as W

PAGE = 128          # rows per page of a paged cache
INTERVAL = 128      # decode steps between two evictions: room for the sentences that these steps open
ROW = 256           # bytes of one bf16 K or V row


def _case(name, op, **over):
    c = dict(name=name, op=op, cache="slab", batch=10, hq=32, hk=8, window=32, d_model=4096, layers=1, lo=2048, hi=2048,
             budget=0, fill=False, lam="keys", sents="uniform", dup=0.3)
    c.update(over)
    return c


def listed():
    return [
        # one user: a decode step of a 32-layer model over a cache of a few thousand tokens; nothing but launches and latency
        _case("step-1seq", "step", batch=1, lo=2048, hi=2048, layers=32),
        # the steady state of the headline workload: ten sequences at the budget of 4096 (a little under, by sentence)
        _case("step-budget4k", "step", lo=4000, hi=4224, layers=2),
        # a paged server with five heads per KV head at the budget of 8192
        _case("step-paged-g5", "step", cache="paged", batch=16, hq=40, window=64, d_model=5120, lo=8000, hi=8320,
              sents="geometric", dup=0.4),
        # decode before any eviction: ragged 16K to 32K contexts
        _case("attn-32k", "attn", lo=16384, hi=32768),
        # an eviction pass on one short sequence, layer by layer
        _case("score-1seq", "score", batch=1, lo=2048, hi=2048, layers=8, dup=0.25),
        # an eviction pass of the decode loop: budget 2048 + 128 new tokens, penalty from the lookup table
        _case("score-loop-table", "score", lo=2113, hi=2176, layers=4, lam="table", dup=0.2),
        # the headline: the first eviction after long prompts, and what follows it
        _case("score-32k", "score", lo=16384, hi=32768),
        _case("evict-32k", "evict", lo=16384, hi=32768, budget=4096),
        # the largest scoring call: 64K contexts, long-tailed sentences, three query blocks per group
        _case("score-64k-g5", "score", batch=16, hq=40, window=64, d_model=5120, lo=32768, hi=65536, sents="geometric",
              dup=0.4),
        # the decode loop's eviction to exactly the budget
        _case("evict-loop-fill", "evict", lo=2113, hi=2176, budget=2048, fill=True, layers=4, dup=0.2),
        # redundancy over single tokens at the budget of 4096 + 128
        _case("token-red-4k", "token_red", lo=4224, hi=4224),
        # every sequence closes a sentence and compares it with those before it
        _case("table-close", "table", lo=1300, hi=1300),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "attn", "score", "score", "evict", "evict", "token_red", "table"])
    hq, hk = rng.choice([(32, 8), (32, 8), (40, 8), (16, 2), (28, 4), (16, 8)])
    batch = _log(rng, 1, 16)
    geo = rng.random() < 0.3
    c = dict(op=op, cache="slab", batch=batch, hq=hq, hk=hk, window=rng.choice([8, 16, 32, 32, 48, 64]),
             d_model=rng.choice([2048, 4096, 5120]), layers=1, lo=0, hi=0, budget=0, fill=False, lam="keys",
             sents="geometric" if geo else "uniform", dup=round(rng.uniform(0.1, 0.5), 2))
    if hq // hk == 7:
        c["window"] = min(c["window"], 48)
    if op == "step":
        c["hi"] = _log(rng, 256, 8400)
        c["cache"] = rng.choice(["slab", "slab", "paged"])
        c["layers"] = rng.choice([1, 2, 4, 8, 16]) if batch * c["hi"] < 20000 else 1
    elif op == "attn":
        c["hi"] = _log(rng, 512, min(65536, 320000 // batch))
        c["cache"] = rng.choice(["slab", "slab", "paged", "static"])
    elif op == "score":
        c["hi"] = _log(rng, 512, min(65536, 400000 // batch))
        c["cache"] = rng.choice(["slab", "slab", "paged"])
        c["lam"] = rng.choice(["keys", "table"]) if c["cache"] == "slab" else "keys"
        c["layers"] = rng.choice([1, 2, 4]) if batch * c["hi"] < 24000 else 1
    elif op == "evict":
        c["hi"] = _log(rng, 512, min(65536, 320000 // batch))
        c["fill"] = rng.random() < 0.4
        c["cache"] = "slab" if c["fill"] else rng.choice(["slab", "slab", "paged"])
        c["layers"] = rng.choice([1, 2, 4]) if batch * c["hi"] < 24000 else 1
    elif op == "token_red":
        c["hi"] = _log(rng, 256, min(8300, int(math.sqrt(1.7e8 / batch))))
        c["lo"] = c["hi"] - rng.randrange(0, 1 + c["hi"] // 16)
    else:
        c["hi"] = _log(rng, 32, 2000)
    if not c["lo"]:
        c["lo"] = max(1, int(c["hi"] * rng.choice([0.5, 0.8, 0.95, 1.0])))
    if op == "evict":
        c["budget"] = max(64, int(c["lo"] * rng.choice([0.125, 0.25, 0.5, 0.94 if batch * c["hi"] < 100000 else 0.3])))
    return c


# ------------------------------------------------------------------------------------------------ sizes
def _tokens(c):
    """Cached tokens of every sequence: evenly spread between lo and hi, long and short ones mixed."""
    n = c["batch"]
    v = np.linspace(c["hi"], c["lo"], n).round().astype(np.int64)
    return v[(np.arange(n) * 7) % n] if n % 7 else v


def _mean_sentence(c):
    return 52.0 if c["sents"] == "uniform" else 24.0


def _max_sent(c):
    """Stride of the sentence tables: what the longest context holds, with some room, and the sentences of one interval."""
    return int(1.25 * c["hi"] / _mean_sentence(c)) + 16 + (INTERVAL if c["op"] == "step" else 0)


def _caps(c):
    """Rows a slab has room for: the cached tokens (+ the new tokens of the interval in a decode loop), whole pages if paged."""
    cap = _tokens(c) + (INTERVAL if c["op"] == "step" else 0)
    return -(-cap // PAGE) * PAGE if c["cache"] == "paged" else cap


def work(case):
    c = case
    hk, n = c["hk"], c["hq"] // c["hk"]
    tok = _tokens(c).astype(float)
    rows = float(tok.sum()) * hk
    L = c["layers"]
    if c["op"] in ("step", "attn"):
        qo = 2.0 * c["batch"] * c["hq"] * ROW + 2.0 * c["batch"] * c["d_model"] * 2
        new = 4.0 * c["batch"] * hk * ROW + c["batch"] * c["hq"] * ROW if c["op"] == "step" else 0.0
        return {"bytes": L * (rows * 2 * ROW + qo + new), "flops": L * rows * n * 128 * 4}
    if c["op"] == "score":
        sent = rows / _mean_sentence(c)
        gram = float(((tok / _mean_sentence(c)) ** 2).sum()) * hk * 128          # symmetric: half of 2 * 128 per entry
        return {"bytes": L * (rows * (ROW + 4) + sent * 5 * 4 + c["batch"] * c["hq"] * c["window"] * ROW),
                "flops": L * (rows * n * c["window"] * 256 + rows * 128 + gram)}
    if c["op"] == "evict":
        kept = float(np.minimum(tok, c["budget"]).sum()) * hk
        sent = rows / _mean_sentence(c)
        return {"bytes": L * (kept * (4 * ROW + 4) + sent * (4 + 2 * 8 + 5)), "flops": 0.0}
    if c["op"] == "token_red":
        return {"bytes": rows * (ROW + 4), "flops": float((tok ** 2).sum()) * hk * 128}
    return {"bytes": float(tok.sum()) * c["d_model"] * 4 + c["batch"] * c["d_model"] * 14, "flops": float(tok.sum()) * c["d_model"] * 2}


def tolerance(case):
    if case["op"] == "evict":
        return "exact"                   # flags, tables and moved rows
    if case["op"] in ("step", "attn"):
        return {"rel": 1e-2}             # bf16 attention output and hidden state
    return {"rel": 1e-5}                 # fp32 sums over bf16 keys (and fp32 embeddings)


# ------------------------------------------------------------------------------------------------ inputs
class _State:
    """What the user's program holds: the caches of all layers (stacked), the tables, outputs and one workspace."""

    def per_layer(self, *names):
        """Under each name, the stacked tensor's layers as a list; the stacked tensor stays under name_all."""
        for name in names:
            t = getattr(self, name)
            setattr(self, name + "_all", t)
            setattr(self, name, list(t.unbind(0)) if t is not None else None)


def _workload(c, seed):
    uni = c["sents"] == "uniform"
    return W.Workload("case", seed, c["batch"], c["hq"], c["hk"], 128, c["window"], c["d_model"], c["budget"], c["lo"], c["hi"],
                      8 if uni else 4, 96 if uni else 128, c["sents"], 20.0, c["dup"], 0.05)


def _make_cache(c, s, g, sents, values=True):
    """K (near-duplicate sentences are noisy copies of their source) and V of every layer; rows past the live ones are noise too."""
    cap, tok, hk, L = _caps(c), _tokens(c), c["hk"], c["layers"]
    off = np.concatenate([[0], np.cumsum(cap)])
    s.rows = int(off[-1]) * hk
    s.K = torch.randn(L, s.rows, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    s.V = torch.randn(L, s.rows, 128, generator=g, device="cuda", dtype=torch.bfloat16) if values else None
    if sents is not None:
        for b, (lengths, src) in enumerate(sents):
            root = np.arange(len(src))
            for i in np.nonzero(src >= 0)[0]:
                root[i] = root[src[i]]
            start = np.concatenate([[0], np.cumsum(lengths)])[:-1]
            delta = np.repeat(start[root] - start, lengths)
            at = np.nonzero(delta)[0]
            if not len(at):
                continue
            dst = torch.from_numpy(at).cuda()
            frm = torch.from_numpy(at + delta[at]).cuda()
            slab = s.K[:, int(off[b]) * hk:int(off[b + 1]) * hk].view(L, hk, int(cap[b]), 128)
            for layer in range(L):
                noise = torch.randn(hk, len(at), 128, generator=g, device="cuda", dtype=torch.bfloat16)
                slab[layer][:, dst] = slab[layer][:, frm].add_(noise, alpha=0.05)
    s.slab_off = torch.from_numpy(off[:-1].copy()).cuda()
    s.cap = torch.from_numpy(cap.astype(np.int32)).cuda()
    s.max_cap = int(cap.max())
    s.kv = np.repeat(tok[:, None], hk, axis=1).astype(np.int32)
    if c["cache"] == "paged":                              # the same number of rows as pages in random order
        s.max_pages = s.max_cap // PAGE
        pages = torch.randperm(s.rows // PAGE, generator=g, device="cuda").to(torch.int32)
        table = torch.zeros(c["batch"], hk, s.max_pages, dtype=torch.int32, device="cuda")
        at = 0
        for b in range(c["batch"]):
            k = int(cap[b]) // PAGE
            table[b, :, :k] = pages[at:at + hk * k].view(hk, k)
            at += hk * k
        s.block_table = table


def _make_tables(c, s, sents):
    """Cache-space range lists of one layer, as one buffer: sent_off, sent_id, n_sent and kv_len are views of it."""
    bt, hk = c["batch"], c["hk"]
    s.max_sent = ms = _max_sent(c)
    off, ids = np.zeros((bt, hk, ms + 1), np.int32), np.full((bt, hk, ms), -1, np.int32)
    n = np.zeros((bt, hk), np.int32)
    for b, (lengths, _) in enumerate(sents):
        k = min(len(lengths), ms)                          # a full list: the rest joins the last sentence
        off[b, :, 1:k + 1] = np.cumsum(lengths)[:k]
        off[b, :, k] = lengths.sum()
        off[b, :, k + 1:] = off[b, :, k:k + 1]
        ids[b, :, :k] = np.arange(k)
        n[b] = k
    s.tables0 = torch.from_numpy(np.concatenate([off.ravel(), ids.ravel(), n.ravel(), s.kv.ravel()])).cuda()
    s.tables = s.tables0.repeat(c["layers"], 1)
    s.off_shape, s.id_shape = off.shape, ids.shape
    return [_views(s, s.tables[layer]) for layer in range(c["layers"])]


def _views(s, flat):
    bt, hk, ms1 = s.off_shape
    a, b = bt * hk * ms1, bt * hk * (ms1 - 1)
    return (flat[:a].view(s.off_shape), flat[a:a + b].view(s.id_shape), flat[a + b:a + b + bt * hk].view(bt, hk),
            flat[a + b + bt * hk:].view(bt, hk))


def _make_shape(c, s, max_sent):
    s.shape = B.make_shape(c["batch"], c["hq"], c["hk"], 128, c["window"], c["d_model"], max_sent, s.max_cap, s.slab_off, s.cap, s.rows)
    s.params = B.make_params(0.1, 0.95, 1e-6, c["budget"], c["window"])
    s.ws = torch.empty(B.skipkv_workspace_bytes(s.shape), dtype=torch.uint8, device="cuda")
    B.skipkv_workspace_init(s.shape, s.ws)


def _make_attention(c, s, g):
    r = lambda *shape: torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    L, bt, hq, hk = c["layers"], c["batch"], c["hq"], c["hk"]
    s.q, s.out = r(L, bt, hq, 128), torch.zeros(L, bt, hq, 128, dtype=torch.bfloat16, device="cuda")
    s.hidden, s.steer = r(L, bt, c["d_model"]), r(c["d_model"]) * 0.01
    s.alpha = 1.0 + 0.02 * torch.randint(0, 40, (bt,), generator=g, device="cuda").float()
    s.flag = (torch.rand(bt, generator=g, device="cuda") < 0.6).to(torch.uint8)
    s.k_new, s.v_new = r(L, bt, hk, 128), r(L, bt, hk, 128)


_STACKED = {"step": ("q", "out", "hidden", "k_new", "v_new", "kv_out", "q_win"), "attn": ("q", "out", "hidden"),
            "score": ("q_win", "tok_imp", "imp", "red", "lam_out", "score"), "token_red": (),
            "evict": ("score", "keep", "kept_idx", "n_kept", "new_len", "index_map")}


def prepare(case, seed):
    c, s = case, _State()
    g = torch.Generator(device="cuda").manual_seed(seed)
    s.op, s.cache, s.fill, s.lam, s.layers = c["op"], c["cache"], c["fill"], c["lam"], range(c["layers"])
    bt, hk, ctx = c["batch"], c["hk"], _tokens(c)
    if c["op"] == "table":
        return _prepare_table(c, s, g, ctx)
    sents = None
    if c["op"] in ("step", "score", "evict"):
        wl = _workload(c, seed)
        sents = [W.draw_sentences(wl, 0, b, int(ctx[b])) for b in range(bt)]
    _make_cache(c, s, g, sents if c["op"] == "score" else None, values=c["op"] not in ("score", "token_red"))
    if sents is not None:
        s.tab = _make_tables(c, s, sents)
    else:
        s.kv_len = torch.from_numpy(s.kv).cuda()
    _make_shape(c, s, s.max_sent if sents is not None else 1)
    f32 = dict(dtype=torch.float32, device="cuda")
    if c["op"] in ("step", "attn"):
        _make_attention(c, s, g)
        if c["op"] == "step":
            s.kv_out = torch.zeros(c["layers"], bt, hk, dtype=torch.int32, device="cuda")
            s.q_win = torch.randn(c["layers"], bt, c["hq"], c["window"], 128, generator=g, device="cuda", dtype=torch.bfloat16)
            s.opens = torch.zeros(bt, dtype=torch.uint8, device="cuda")          # the token continues a sentence, as most do
            s.gen_id = torch.full((bt,), s.max_sent, dtype=torch.int32, device="cuda")
            s.slot = seed % c["window"]
    elif c["op"] == "score":
        L, slab_rows = c["layers"], s.max_pages * PAGE * bt * hk if c["cache"] == "paged" else s.rows
        s.q_win = torch.randn(L, bt, c["hq"], c["window"], 128, generator=g, device="cuda", dtype=torch.bfloat16)
        s.tok_imp = torch.zeros(L, slab_rows, **f32)
        s.imp, s.red, s.lam_out, s.score = (torch.zeros(L, bt, hk, s.max_sent, **f32) for _ in range(4))
        if c["lam"] == "table":                                                  # the table that the decode steps kept
            sim = 0.95 + 0.05 * torch.rand(bt, s.max_sent, generator=g, **f32)
            s.lam_table = torch.where(torch.rand(bt, s.max_sent, generator=g, **f32) < c["dup"], sim, torch.zeros_like(sim))
    elif c["op"] == "evict":
        # scores as the scoring call leaves them: minus one over the number of sentences, spread by importance, and about
        # one below that for the sentences that a later one repeats
        L, cnt = c["layers"], torch.tensor([len(x[0]) for x in sents], device="cuda").view(1, bt, 1, 1)
        base = -0.9 / cnt + 2e-4 * torch.randn(L, bt, hk, s.max_sent, generator=g, **f32)
        lam = 0.95 + 0.05 * torch.rand(L, bt, hk, s.max_sent, generator=g, **f32)
        s.score = base - torch.where(torch.rand(L, bt, hk, s.max_sent, generator=g, **f32) < c["dup"], lam, torch.zeros_like(lam))
        s.keep = torch.zeros(L, bt, hk, s.max_sent, dtype=torch.uint8, device="cuda")
        s.kept_idx = torch.zeros(L, bt, hk, s.max_sent, dtype=torch.int32, device="cuda")
        s.n_kept, s.new_len = (torch.zeros(L, bt, hk, dtype=torch.int32, device="cuda") for _ in range(2))
        map_rows = s.max_pages * PAGE * bt * hk if c["cache"] == "paged" else s.rows
        s.index_map = torch.full((L, map_rows), -1, dtype=torch.int32, device="cuda")
        if c["fill"]:
            s.tok_imp = torch.rand(L, s.rows, generator=g, **f32) * (2.0 / c["hi"])
            s.tok_keep = torch.zeros(L, s.rows, dtype=torch.uint8, device="cuda")
    else:
        s.tok_red = torch.zeros(s.rows, **f32)
    s.per_layer("K", "V", *_STACKED[c["op"]], *(("tok_imp", "tok_keep") if c["fill"] else ()))
    return s


def _prepare_table(c, s, g, ctx):
    """Unit embeddings of the earlier sentences (two of them close to the one that is about to close) and its running sum."""
    bt, dm = c["batch"], c["d_model"]
    s.bt, s.dm, s.mg = bt, dm, int(ctx.max()) + 64
    s.emb = torch.randn(bt, s.mg, dm, generator=g, device="cuda")
    s.hidden = torch.randn(bt, dm, generator=g, device="cuda").bfloat16()
    for k, spread in ((2, 0.1), (3, 0.2)):
        rows = torch.from_numpy(ctx // k).cuda()
        noise = torch.randn(bt, dm, generator=g, device="cuda")
        s.emb[torch.arange(bt, device="cuda"), rows] = s.hidden.float() + spread * noise
    s.emb /= s.emb.norm(dim=-1, keepdim=True) + 1e-6
    s.acc = 20 * s.hidden.float() + 2 * torch.randn(bt, dm, generator=g, device="cuda")
    s.acc_count = torch.full((bt,), 20, dtype=torch.int32, device="cuda")
    s.flag = torch.ones(bt, dtype=torch.uint8, device="cuda")
    s.n0 = torch.from_numpy(ctx.astype(np.int32)).cuda()
    s.n_gen, s.closed = s.n0.clone(), torch.zeros(bt, dtype=torch.int32, device="cuda")
    s.lam_table = torch.zeros(bt, s.mg, device="cuda")
    s.status = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ the calls
def run(s):
    if s.op == "step":
        # the lengths go from one buffer to another; a loop swaps the two, here every pass appends the same token
        for i in s.layers:
            so, sid, ns, kv = s.tab[i]
            if s.cache == "paged":
                B.skipkv_decode_step_paged(s.shape, s.q[i], s.k_new[i], s.v_new[i], s.K[i], s.V[i], s.block_table, s.max_pages, kv,
                                           s.kv_out[i], so, sid, ns, s.opens, s.gen_id, s.q_win[i], s.slot, s.out[i], s.hidden[i],
                                           s.steer, s.alpha, s.flag, s.ws)
            else:
                B.skipkv_decode_step(s.shape, s.q[i], s.k_new[i], s.v_new[i], s.K[i], s.V[i], kv, s.kv_out[i], so, sid, ns, s.opens,
                                     s.gen_id, s.q_win[i], s.slot, s.out[i], s.hidden[i], s.steer, s.alpha, s.flag, s.ws)
        return {"out": s.out_all, "hidden": s.hidden_all, "K": s.K_all, "V": s.V_all, "kv_len": s.kv_out_all, "tables": s.tables,
                "q_win": s.q_win_all}
    if s.op == "attn":
        for i in s.layers:
            if s.cache == "paged":
                B.skipkv_decode_attn_paged(s.shape, s.q[i], s.K[i], s.V[i], s.block_table, s.max_pages, s.kv_len, s.out[i],
                                           s.hidden[i], s.steer, s.alpha, s.flag, s.ws)
            elif s.cache == "static":
                B.skipkv_decode_attn_static(s.shape, s.q[i], s.K[i], s.V[i], s.kv_len, s.out[i], s.hidden[i], s.steer, s.alpha, s.flag)
            else:
                B.skipkv_decode_attn(s.shape, s.q[i], s.K[i], s.V[i], s.kv_len, s.out[i], s.hidden[i], s.steer, s.alpha, s.flag, s.ws)
        return {"out": s.out_all, "hidden": s.hidden_all}
    if s.op == "score":
        for i in s.layers:
            so, sid, ns, kv = s.tab[i]
            outs = (s.tok_imp[i], s.imp[i], s.red[i], s.lam_out[i], s.score[i])
            if s.lam == "table":
                B.skipkv_score_table(s.shape, s.params, s.K[i], s.q_win[i], kv, so, sid, ns, s.lam_table, s.max_sent, *outs, s.ws)
            elif s.cache == "paged":
                B.skipkv_score_paged(s.shape, s.params, s.K[i], s.block_table, s.max_pages, s.q_win[i], kv, so, ns, *outs, s.ws)
            else:
                B.skipkv_score(s.shape, s.params, s.K[i], s.q_win[i], kv, so, ns, *outs, s.ws)
        return {"tok_imp": s.tok_imp_all, "imp": s.imp_all, "red": s.red_all, "lam": s.lam_out_all, "score": s.score_all}
    if s.op == "evict":
        # the tables as the decode steps left them: compaction rewrites them in place, so every pass starts from a copy
        s.tables.copy_(s.tables0)
        for i in s.layers:
            so, sid, ns, kv = s.tab[i]
            if s.fill:
                B.skipkv_select_fill(s.shape, s.params, s.score[i], s.tok_imp[i], so, ns, s.keep[i], s.tok_keep[i], s.kept_idx[i],
                                     s.n_kept[i], s.new_len[i], s.ws)
                B.skipkv_compact_fill(s.shape, s.K[i], s.V[i], s.keep[i], s.tok_keep[i], so, sid, ns, kv, s.index_map[i], s.ws)
                continue
            B.skipkv_select(s.shape, s.params, s.score[i], so, ns, s.keep[i], s.kept_idx[i], s.n_kept[i], s.new_len[i], s.ws)
            if s.cache == "paged":
                B.skipkv_compact_paged(s.shape, s.K[i], s.V[i], s.block_table, s.max_pages, s.keep[i], so, sid, ns, kv, s.index_map[i],
                                       s.ws)
            else:
                B.skipkv_compact(s.shape, s.K[i], s.V[i], s.keep[i], so, sid, ns, kv, s.index_map[i], s.ws)
        return {"keep": s.keep_all, "kept_idx": s.kept_idx_all, "n_kept": s.n_kept_all, "new_len": s.new_len_all, "tables": s.tables,
                "index_map": s.index_map_all, "K": s.K_all, "V": s.V_all}
    if s.op == "token_red":
        B.skipkv_token_redundancy(s.shape, s.params, s.K[0], s.kv_len, s.tok_red, s.ws)
        return {"tok_red": s.tok_red}
    # the number of sentences as it was before this step: the pass closes the same sentence every time
    s.n_gen.copy_(s.n0)
    B.skipkv_table_step(s.bt, s.dm, s.mg, s.hidden, s.flag, s.acc, s.acc_count, s.emb, s.n_gen, s.closed, s.lam_table, 0.95, 1e-6, s.status)
    return {"emb": s.emb, "lam": s.lam_table, "n": s.n_gen, "closed": s.closed, "acc": s.acc, "count": s.acc_count, "status": s.status}
