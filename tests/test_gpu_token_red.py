"""GPU parity of the token-level redundancy term (skipkv_token_redundancy) against the CPU oracle:
every live row of every slab, rtol 1e-3 (fp32 dot products of exact bf16 products, one approximate
exponential per matrix element), plus the invariant that a slab's values sum to 1."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_07993_b200 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "smoke": lambda: W.config(0),
    "ragged": lambda: W.config(0, batch=3, ctx_lo=100, ctx_hi=1500, budget=256, seed=77),
    "one-tile": lambda: W.config(0, batch=2, ctx_lo=1, ctx_hi=128, seed=80),
    "steady-state": lambda: W.config(0, batch=1, ctx_lo=4224, ctx_hi=4224, sent_lo=8, sent_hi=96, seed=81),
    "spare-rows": lambda: W.config(0, batch=2, ctx_lo=700, ctx_hi=900, cap_extra=77, seed=82),
}


def run(cfg, kv_len_override=None):
    from paper_2512_07993_b200 import build, binding as B
    build.build()
    L = W.make_layer(cfg)
    if kv_len_override is not None:
        L["kv_len"] = kv_len_override(L["kv_len"].copy())
    D = B.DeviceLayer(L)
    red = torch.full((D.K.shape[0],), float("nan"), dtype=torch.float32, device="cuda")
    B.skipkv_token_redundancy(D.shape, D.params, D.K, D.kv_len, red, D.ws)
    torch.cuda.synchronize()
    assert D.status() == 0
    return L, red.cpu().numpy()


@pytest.mark.parametrize("case", list(CASES))
def test_token_redundancy_parity(case):
    cfg = CASES[case]()
    L, red = run(cfg)
    Kb = W.bf16_bits(L["K"])
    for b in range(cfg.batch):
        for h in range(cfg.n_kv_heads):
            rows = W.slab_rows(L, b, h)
            N = int(L["kv_len"][b, h])
            ref = oracle.token_redundancy(Kb[rows][:N], 1e-6)
            got = red[rows][:N].astype(np.float64)
            err = np.abs(got - ref) - 1e-3 * np.abs(ref)
            assert (err <= 0).all(), f"slab ({b},{h}): worst excess {err.max():.3e} at {int(err.argmax())} of {N}"
            if N > 1:
                assert abs(got.sum() - 1.0) < 1e-3
            assert np.isnan(red[rows][N:]).all()            # rows beyond the live ones are not written


def test_token_redundancy_empty_and_single_row_slabs():
    cfg = CASES["smoke"]()
    def override(kv):
        kv[0, 0] = 0; kv[0, 1] = 1; kv[1, 0] = 129
        return kv
    L, red = run(cfg, override)
    Kb = W.bf16_bits(L["K"])
    for b in range(cfg.batch):
        for h in range(cfg.n_kv_heads):
            rows = W.slab_rows(L, b, h)
            N = int(L["kv_len"][b, h])
            got = red[rows]
            assert np.isnan(got[N:]).all()
            if N == 1:
                assert got[0] == 0.0
            elif N > 1:
                ref = oracle.token_redundancy(Kb[rows][:N], 1e-6)
                assert (np.abs(got[:N] - ref) <= 1e-3 * np.abs(ref)).all()


def test_token_redundancy_with_more_slabs_than_shared_memory_has_room_for():
    """9216 slabs: the kernels' table of slabs is in global memory.  Slabs of no row, of one, of whole and partly filled tiles."""
    from paper_2512_07993_b200 import build, binding as B
    build.build()
    lens = np.tile([0, 1, 2, 127, 128, 129, 300, 31, 5], 16)
    bt, hk = len(lens), 64
    off = np.concatenate([[0], np.cumsum(lens)])
    g = torch.Generator(device="cuda").manual_seed(83)
    K = torch.randn(int(off[-1]) * hk, 128, generator=g, device="cuda").bfloat16()
    slab_off, cap = torch.as_tensor(off[:-1].copy()).cuda(), torch.as_tensor(lens.astype(np.int32)).cuda()
    shape = B.make_shape(bt, hk, hk, 128, 8, 0, 1, int(lens.max()), slab_off, cap, K.shape[0])
    ws = torch.empty(B.skipkv_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    B.skipkv_workspace_init(shape, ws)
    kv_len = cap[:, None].repeat(1, hk).contiguous()
    red = torch.full((K.shape[0],), float("nan"), device="cuda")
    B.skipkv_token_redundancy(shape, B.make_params(), K, kv_len, red, ws)
    torch.cuda.synchronize()
    assert B.skipkv_status(ws) == 0
    for b in range(bt):
        n = int(lens[b])
        if n == 0:
            continue
        got = red[off[b] * hk:off[b + 1] * hk].view(hk, n)
        k = K[off[b] * hk:off[b + 1] * hk].view(hk, n, 128).double()
        k = k / (k.norm(dim=-1, keepdim=True) + 1e-6)
        e = torch.exp(k @ k.transpose(1, 2)) * (1 - torch.eye(n, device="cuda", dtype=torch.float64))
        ref = (e / e.sum(-1, keepdim=True).clamp_min(1e-30)).sum(1) / n
        assert ((got - ref).abs() <= 1e-3 * ref.abs()).all(), b


@pytest.mark.parametrize("ctx,hk", [(4224, 4), (7611, 2), (300, 4)])
def test_token_redundancy_is_rounded_once(ctx, hk):
    """Error against 64 bits (2-norm): the result's own rounding (2^-24 / sqrt 3 = 3.4e-8), the means over thousands of terms add nothing to speak of.
    Sums that grow to their full size by one reduction after the other are off by 8.6e-8 at 4224 rows and 1.3e-7 at 7611."""
    cfg = W.config(0, batch=1, n_q_heads=hk, n_kv_heads=hk, ctx_lo=ctx, ctx_hi=ctx, sent_lo=8, sent_hi=96, seed=84)
    L, red = run(cfg)
    for h in range(hk):
        rows = W.slab_rows(L, 0, h)
        k = L["K"][rows].cuda().double()
        k = k / (k.norm(dim=-1, keepdim=True) + 1e-6)
        e = torch.exp(k @ k.T).fill_diagonal_(0)
        ref = (e / e.sum(-1, keepdim=True)).sum(0) / ctx
        err = (torch.as_tensor(red[rows]).cuda().double() - ref).norm() / ref.norm()
        assert err <= 5e-8, (h, float(err))
