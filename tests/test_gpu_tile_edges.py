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
