"""Sizes at the edges of the kernels' tiles, on every branch of their dispatch, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_07993_b200 import workloads as W

pytestmark = pytest.mark.gpu


def layer(ctx, **over):
    from paper_2512_07993_b200 import build, binding as B
    build.build()
    cfg = W.config(0, batch=len(ctx), ctx_lo=min(ctx), ctx_hi=max(ctx), **over)
    L = W.make_layer(cfg, ctx=np.asarray(ctx))
    return B, L, B.DeviceLayer(L)


def oshape(L):
    cfg = L["cfg"]
    return dict(batch=cfg.batch, Hq=cfg.n_q_heads, Hk=cfg.n_kv_heads, d=cfg.head_dim, alpha=cfg.window,
                max_sent=L["max_sent"], slab_off=L["slab_off"], cap=L["cap"])


@pytest.mark.parametrize("hq", [2, 4, 6, 8, 10, 12, 14, 16])
def test_decode_rows_around_warp_and_tile_edges(hq):
    """16 rows per warp, 64 per tile: lengths on both sides of each edge, one to eight heads per KV head, fewer and more
    tiles than CTAs."""
    for ctx in ([1, 2, 15, 16, 17, 31, 33, 48, 49], [63, 64, 65, 127, 128, 129, 191], [6000, 5951, 6081]):
        B, L, D = layer(ctx, n_q_heads=hq, n_kv_heads=2, seed=300 + hq, cap_extra=1)
        for t in (D.K, D.V):                              # rows past the live ones must not matter
            for b in range(len(ctx)):
                for h in range(2):
                    t[W.slab_rows(L, b, h)][int(L["kv_len"][b, h]):] = float("nan")
        D.out.fill_(float("nan"))
        D.decode_attn(steer=False)
        torch.cuda.synchronize()
        assert D.status() == 0
        _, o64 = oracle.decode_attn_batch(oshape(L), W.bf16_bits(L["q"]), W.bf16_bits(L["K"]), W.bf16_bits(L["V"]), L["kv_len"])
        out = D.out.float().cpu().numpy().astype(np.float64)
        err = np.abs(out - o64) / np.abs(o64).max(axis=-1, keepdims=True)
        assert np.isfinite(out).all() and err.max() <= 2e-2 and np.sqrt((err ** 2).mean()) < 2e-3


@pytest.mark.parametrize("step", [False, True])
def test_decode_reads_every_row_whatever_total_rows_says(step):
    """total_rows bounds the copies that go out before the lengths are confirmed.  With one that ends behind a slab whose last tile is the first
    of a CTA's share, that CTA's second tile lies beyond it and is copied behind the confirmation: the same bits as with the true number."""
    ctx = [1300 + 171 * i for i in range(12)]
    B, L, D = layer(ctx, n_q_heads=8, n_kv_heads=2, seed=340, cap_extra=1)
    tiles = np.repeat([(n + step + 63) // 64 for n in ctx], 2)
    ends, rows_end = np.cumsum(tiles), np.cumsum(np.repeat([n + 1 for n in ctx], 2))
    ctas = min(torch.cuda.get_device_properties(0).multi_processor_count, 256, int(ends[-1]))
    starts = [c * int(ends[-1]) // ctas for c in range(ctas)]
    short = [int(rows_end[s]) for s in range(23) if ends[s] - 1 in starts]
    assert short
    cfg = L["cfg"]
    row = lambda seed: torch.randn(12, 2, 128, generator=torch.Generator().manual_seed(seed)).bfloat16().cuda()
    one = lambda dt, v: torch.full((12,), v, dtype=dt, device="cuda")

    def run(total_rows):
        shp = B.make_shape(12, 8, 2, 128, cfg.window, cfg.d_model, D.max_sent, max(ctx) + 1, D.slab_off, D.cap, total_rows)
        out = torch.full_like(D.out, float("nan"))
        if step:
            B.skipkv_decode_step(shp, D.q, row(1), row(2), D.K.clone(), D.V.clone(), D.kv_len, torch.empty_like(D.kv_len), D.sent_off.clone(),
                                 D.sent_id.clone(), D.n_sent.clone(), one(torch.uint8, 0), one(torch.int32, 0), None, 0, out, None, None, None, None, D.ws)
        else:
            B.skipkv_decode_attn(shp, D.q, D.K, D.V, D.kv_len, out, None, None, None, None, D.ws)
        torch.cuda.synchronize()
        assert D.status() == 0
        return out

    want = run(int(D.K.shape[0]))
    for total_rows in short:
        assert torch.equal(run(total_rows).view(torch.int16), want.view(torch.int16)), total_rows


def check_scores(B, L, D, rtol=1e-3):
    cfg = L["cfg"]
    D.score()
    torch.cuda.synchronize()
    assert D.status() == 0
    ref = oracle.score_batch(oshape(L), W.bf16_bits(L["K"]), W.bf16_bits(L["q_win"]), L["kv_len"], L["sent_off"], L["n_sent"],
                             float(np.float32(0.1)), float(np.float32(0.95)), float(np.float32(1e-6)), want_tok_imp=True)
    live = np.arange(L["max_sent"])[None, None, :] < L["n_sent"][:, :, None]
    for name, got in (("imp", D.sent_imp), ("red", D.sent_red), ("lam", D.sent_lam), ("score", D.sent_score)):
        g, r = got.cpu().numpy()[live].astype(np.float64), np.asarray(ref[name], np.float64)[live]
        assert (np.abs(g - r) <= rtol * np.abs(r) + 1e-7).all(), (name, np.abs(g - r).max())
    tok = D.tok_imp.cpu().numpy()
    for b in range(cfg.batch):
        for h in range(cfg.n_kv_heads):
            rows = W.slab_rows(L, b, h)
            n = int(L["kv_len"][b, h])
            g, r = tok[rows][:n].astype(np.float64), np.asarray(ref["tok_imp"], np.float64)[rows][:n]
            assert (np.abs(g - r) <= rtol * np.abs(r)).all(), ("tok_imp", b, h)


@pytest.mark.parametrize("sentences", [[1, 2, 31, 33], [63, 64, 65, 128], [127, 129, 5, 1], [256, 257, 300], [640, 1153], [4225]])
def test_score_sentence_counts_around_a_tile(sentences):
    """Up to 128 sentences per slab: one kernel behind the sweeps; more: the blocked kernels, block columns cut by the CTAs' ranges
    or not, and partial sums that outgrow the key sums."""
    B, L, D = layer([5 * n for n in sentences], sent_lo=5, sent_hi=5, dup_rate=0.3, seed=500 + sentences[0])
    assert int(L["n_sent"].max()) == max(sentences)
    check_scores(B, L, D)


@pytest.mark.parametrize("group,window", [(1, 1), (1, 16), (1, 17), (1, 127), (1, 512), (2, 33), (2, 128), (3, 32), (3, 128), (4, 31),
                                          (4, 96), (5, 17), (5, 64), (6, 16), (6, 64), (7, 48), (7, 72), (8, 15), (8, 49)])
def test_score_query_blocks(group, window):
    """Blocks of 32 and of 16 window positions, one to sixteen of them, one and several per row operand, whole and partly
    filled; slabs of less than a tile, of whole tiles and of many tiles in one CTA's share."""
    for ctx in ([100, 128, 129, 520], [4100, 9000, 257, 128]):
        B, L, D = layer([max(c, window) for c in ctx], n_q_heads=2 * group, n_kv_heads=2, window=window, sent_lo=8, sent_hi=40,
                        dup_rate=0.3, seed=700 + 10 * group + window % 10)
        check_scores(B, L, D)


@pytest.mark.parametrize("group,window", [(4, 32), (5, 64), (4, 48)])
@pytest.mark.parametrize("lo,hi", [(9000, 9000), (700, 3000), (127, 129), (3, 20000)])
def test_score_sentences_across_the_ranges_of_several_ctas(group, window, lo, hi):
    """A sentence's key sum comes from every CTA that has some of its tokens: sentences of one token up to whole slabs over many CTAs, empty
    ones between them, starts on and beside tile edges; with the sums in either pass (one operand of query rows, several)."""
    ctx = [40000, 9000, 130]
    B, L, D = layer(ctx, n_q_heads=2 * group, n_kv_heads=2, window=window, sent_lo=8, sent_hi=12, dup_rate=0.3, seed=760 + group)
    rng = np.random.Generator(np.random.Philox(lo))
    for b, n in enumerate(ctx):
        at = [0]
        while at[-1] < n:
            step = lo if lo == hi else int(np.exp(rng.uniform(np.log(lo), np.log(hi))))
            at.append(min(at[-1] + step, n))
            if rng.random() < 0.1:
                at.append(at[-1])                         # an empty sentence
            if len(at) > L["max_sent"]:
                at = at[:L["max_sent"]] + [n]
                break
        S = len(at) - 1
        L["sent_off"][b, :, :S + 1] = at
        L["sent_off"][b, :, S + 1:] = n
        L["n_sent"][b] = S
    D.sent_off.copy_(torch.from_numpy(np.ascontiguousarray(L["sent_off"])))
    D.n_sent.copy_(torch.from_numpy(np.ascontiguousarray(L["n_sent"])))
    check_scores(B, L, D)


@pytest.mark.parametrize("group,window,batch,sent", [(1, 512, 16, (8, 40)), (5, 100, 19, (8, 40)), (1, 512, 16, (2, 4))])
def test_score_with_more_slabs_than_shared_memory_has_room_for(group, window, batch, sent):
    """Over a thousand slabs beside a wide window: the sweep's table of slabs is in global memory; contiguous against the oracle, paged
    against contiguous, up to 128 sentences per slab and more."""
    lens = [1, 2, 127, 128, 129, 255, 256, 257, 384, 40, 77, 300, 500, 9, 16, 130, 31, 64, 200][:batch]
    B, L, D = layer(lens, n_q_heads=64 * group, n_kv_heads=64, window=window, sent_lo=sent[0], sent_hi=sent[1], dup_rate=0.3, seed=900 + group)
    assert batch * 64 > 1000 and (int(L["n_sent"].max()) > 128) == (sent[1] < 8)
    check_scores(B, L, D)
    pages = -(-np.asarray(lens) // 128)
    max_pages, n_pool = int(pages.max()), int(pages.sum()) * 64
    ids = np.random.Generator(np.random.Philox(5)).permutation(n_pool)
    Kp = torch.full((n_pool * 128, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    table, k = np.full((batch, 64, max_pages), -1, np.int32), 0
    for b in range(batch):
        for h in range(64):
            table[b, h, :pages[b]] = ids[k:k + pages[b]]
            k += pages[b]
    table = torch.as_tensor(table).cuda()
    for b, n in enumerate(lens):
        t = torch.arange(n, device="cuda")
        rows = table[b].long()[:, t // 128] * 128 + t % 128
        off = int(L["slab_off"][b]) * 64
        Kp[rows.reshape(-1)] = D.K[off:off + 64 * n]
    shp = B.make_shape(batch, 64 * group, 64, 128, window, L["cfg"].d_model, D.max_sent, max(lens), D.slab_off, D.cap, int(Kp.shape[0]))
    imp = torch.full((batch, 64, max_pages * 128), float("nan"), device="cuda")
    outs = [torch.full_like(D.sent_imp, float("nan")) for _ in range(4)]
    B.skipkv_score_paged(shp, D.params, Kp, table, max_pages, D.q_win, D.kv_len, D.sent_off, D.n_sent, imp, *outs, D.ws)
    torch.cuda.synchronize()
    assert D.status() == 0
    for b, n in enumerate(lens):
        off, S = int(L["slab_off"][b]) * 64, int(L["n_sent"][b, 0])
        assert torch.equal(imp[b, :, :n].reshape(-1), D.tok_imp[off:off + 64 * n])
        for got, ref in zip(outs, (D.sent_imp, D.sent_red, D.sent_lam, D.sent_score)):
            assert torch.equal(got[b, :, :S], ref[b, :, :S])


@pytest.mark.parametrize("group,window,batch", [(1, 512, 14), (4, 128, 15), (6, 84, 6)])
def test_score_with_shared_memory_nearly_full_of_slabs(group, window, batch):
    """The table of slabs beside 512 rows of query operands and one tile stage: 896 slabs (room for 948), 960, and 384 (room for 436) with a short
    last block of rows, whose sums of shifted tiles lie behind the others'."""
    lens = [1, 2, 127, 128, 129, 255, 256, 257, 384, 40, 77, 300, 500, 9, 16][:batch]
    B, L, D = layer(lens, n_q_heads=64 * group, n_kv_heads=64, window=window, sent_lo=8, sent_hi=40, dup_rate=0.3, seed=930 + group)
    check_scores(B, L, D)


@pytest.mark.parametrize("group,window", [(4, 32), (5, 20), (8, 16), (4, 48)])
@pytest.mark.parametrize("ctx", [[1 + (37 * i) % 128 for i in range(64)], [9000, 100, 9000], [9000, 100, 128, 1, 9000]])
def test_score_runs_of_slabs_of_one_tile(group, window, ctx):
    """Three and more slabs of one tile one after the other in a CTA's share, each with one product of the second pass (48 positions: two): short
    sequences throughout, and the eight heads of one or a few among long ones.  The epilogue group that prepares a slab's log-sum-exps is then
    another one every time, and two slabs ahead of the product before.  Contiguous against the oracle, paged against contiguous."""
    B, L, D = layer(ctx, n_q_heads=8 * group, n_kv_heads=8, window=window, sent_lo=8, sent_hi=40, dup_rate=0.3, seed=980 + group)
    check_scores(B, L, D)
    pages = [-(-n // 128) for n in ctx]
    max_pages, n_pool = max(pages), 8 * sum(pages)
    ids = torch.as_tensor(np.random.Generator(np.random.Philox(6)).permutation(n_pool).astype(np.int32)).cuda()
    Kp = torch.full((n_pool * 128, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    table = torch.full((len(ctx), 8, max_pages), -1, dtype=torch.int32, device="cuda")
    k = 0
    for b, n in enumerate(ctx):
        table[b, :, :pages[b]] = ids[k:k + 8 * pages[b]].view(8, pages[b])
        k += 8 * pages[b]
        t = torch.arange(n, device="cuda")
        off = int(L["slab_off"][b]) * 8
        Kp[(table[b].long()[:, t // 128] * 128 + t % 128).reshape(-1)] = D.K[off:off + 8 * n]
    shp = B.make_shape(len(ctx), 8 * group, 8, 128, window, L["cfg"].d_model, D.max_sent, max(ctx), D.slab_off, D.cap, int(Kp.shape[0]))
    imp = torch.full((len(ctx), 8, max_pages * 128), float("nan"), device="cuda")
    outs = [torch.full_like(D.sent_imp, float("nan")) for _ in range(4)]
    B.skipkv_score_paged(shp, D.params, Kp, table, max_pages, D.q_win, D.kv_len, D.sent_off, D.n_sent, imp, *outs, D.ws)
    torch.cuda.synchronize()
    assert D.status() == 0
    for b, n in enumerate(ctx):
        off, S = int(L["slab_off"][b]) * 8, int(L["n_sent"][b, 0])
        assert torch.equal(imp[b, :, :n].reshape(-1), D.tok_imp[off:off + 8 * n])
        for got, ref in zip(outs, (D.sent_imp, D.sent_red, D.sent_lam, D.sent_score)):
            assert torch.equal(got[b, :, :S], ref[b, :, :S])


@pytest.mark.parametrize("hq,ctx", [(2, [30000, 23456]), (8, [4100, 9000, 20000]), (10, [16384, 8000]), (16, [2048, 12345])])
def test_decode_keeps_fp32_probabilities(hq, ctx):
    """The share of outputs that are not the exact result rounded to bf16.  A value with relative error e lies on the wrong side of
    a rounding boundary with probability e times 2^8 (its bf16 ulps), about e * 2^10 on average over outputs that are normal
    around zero.  Probabilities, logits and sums in fp32 (exponential 2 ulp, logits of up to 8 to 2^-22): e < 6e-7, a share of 6e-4;
    probabilities of 16 bits: e = 2^-18, a share of 4e-3."""
    B, L, D = layer(ctx, n_q_heads=hq, n_kv_heads=2, seed=330 + hq)
    wrong = total = 0
    for rep in range(8):
        L["q"] = torch.randn(L["q"].shape, generator=torch.Generator().manual_seed(rep)).bfloat16()
        D.q.copy_(L["q"])
        D.decode_attn(steer=False)
        torch.cuda.synchronize()
        assert D.status() == 0
        for b in range(len(ctx)):
            for h in range(2):
                n = int(L["kv_len"][b, h])
                k, v = (t[W.slab_rows(L, b, h)][:n].double() for t in (D.K, D.V))
                g = slice(h * hq // 2, (h + 1) * hq // 2)
                ref = torch.softmax(D.q[b, g].double() @ k.T / 128 ** 0.5, -1) @ v
                wrong += int((D.out[b, g] != ref.bfloat16()).sum())
                total += ref.numel()
    assert wrong <= 1e-3 * total + 3, (wrong, total)


@pytest.mark.parametrize("group,window,ctx", [(4, 32, [2048, 1500]), (4, 32, [20000, 30011]), (5, 64, [40000]), (8, 16, [700, 9000])])
def test_score_importance_keeps_fp32_logits(group, window, ctx):
    """Error of the token importances against 64 bits (2-norm over a slab's tokens).  A probability 2^x is off by ln 2 times the error of x: a
    logit of up to 32 raw units, truncated a few times at 2^-19, times 0.13 for base 2: 3e-7 at most; its row's log-sum-exp 2^-22; the
    exponential 2^-22 of itself.  The mean over the window's 16 rows and more makes that 1e-7 where the errors of the rows are independent.
    A sum that holds the whole log-sum-exp (120 raw units), or a logarithm of the whole sum (10 and more, to 2^-22 of itself), is off by the
    same amount in all rows: 4e-7 to 9e-7."""
    B, L, D = layer(ctx, n_q_heads=2 * group, n_kv_heads=2, window=window, sent_lo=8, sent_hi=60, seed=950 + group)
    D.score()
    torch.cuda.synchronize()
    assert D.status() == 0
    for b in range(len(ctx)):
        for h in range(2):
            rows, n = W.slab_rows(L, b, h), int(L["kv_len"][b, h])
            k = D.K[rows][:n].double()
            q = D.q_win[b, h * group:(h + 1) * group].double().reshape(group * window, 128)
            ref = torch.softmax(q @ k.T / 128 ** 0.5, -1).view(group, window, n).amax(0).mean(0)
            err = (D.tok_imp[rows][:n].double() - ref).norm() / ref.norm()
            assert err <= 2e-7, (b, h, float(err))
