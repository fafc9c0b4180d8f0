"""A key far above its work item's reference, at columns that each scoring kernel exponentiates on the
FMA pipe (column pairs 3 and 5 of a 32-column chunk) and on the special-function unit (pair 0): the item
must be recomputed and the result must match."""
import numpy as np
import pytest
import torch

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import workloads as wl
import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(16, 16), (32, 64)], ids=["32_rows", "256_rows"])
@pytest.mark.parametrize("col", [0, 7, 10])
def test_out_of_range_column_on_either_pipe(col, H, W):
    ctx = skv.Context(0)
    cfg = wl.PrefillConfig("outlier", B=1, L=8, H=H, Hkv=8, d=64, N=2048, W=W, S=6, shot_dist="uniform", shot_lo=200,
                           shot_hi=400, question_len=100, r_p=0.5, cfg_id=23)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    Q[..., 0], K[..., 0] = 8.0, 0.0
    t = 3 * 128 + 32 + col
    K[0, 0, :, t, 0] = 2000.0                 # logit 8 * 2000 / sqrt(64) = 2000
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    assert skv.shotkv_repaired_items(ctx) == cfg.Hkv
    s = int(np.searchsorted(off[0], t, side="right")) - 1
    k = int(off[0, s + 1] - off[0, s])
    np.testing.assert_allclose(gpu["shot_scores"][0, 0, s].item(), cfg.H * cfg.W / k, rtol=1e-4)
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p)
    ctx.close()


@pytest.mark.parametrize("G,W", [(1, 1), (1, 31), (2, 16), (1, 33), (3, 32), (1, 97), (4, 32), (3, 43), (4, 56), (5, 45), (4, 64)])
def test_token_importance_at_edges_of_32_row_chunks(G, W):
    """Window rows (1, 31, 32, 33, 96, 97, 128, 129, 224, 225, 256) on both sides of the second pass's 32-row
    chunks: chunks without a row are left out."""
    ctx = skv.Context(0)
    cfg = wl.PrefillConfig("chunks", B=1, L=1, H=2 * G, Hkv=2, d=128, N=1411, W=W, S=5, shot_dist="uniform", shot_lo=100,
                           shot_hi=400, question_len=211, r_p=0.5, cfg_id=24)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "calls")
    assert gpu["token_importance"] is not None
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p, check_tokens=True)
    ctx.close()


@pytest.mark.parametrize("d,H,W", [(64, 16, 16), (128, 16, 24), (128, 32, 33), (64, 32, 64)], ids=["32_rows", "48_rows", "132_rows", "256_rows"])
def test_some_of_the_items_of_every_cta_out_of_range(d, H, W):
    """More units than SMs, two layers of every three with a key out of range: a CTA recomputes some of its
    items, of several units, and leaves the others as they are."""
    ctx = skv.Context(0)
    cfg = wl.PrefillConfig("outliers", B=2, L=24, H=H, Hkv=8, d=d, N=1100, W=W, S=4, shot_dist="uniform", shot_lo=150,
                           shot_hi=300, question_len=100, r_p=0.5, cfg_id=25)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    Q[..., 0], K[..., 0] = 8.0, 0.0
    _, chunk_keys, _ = skv.shotkv_plan_pieces(P.dims_of(cfg), off)
    assert chunk_keys >= 256, "the case needs work items of at least two tiles"
    t = min(chunk_keys, 1024) - 128 + 45         # in a later tile of every unit's first item
    marked = [l for l in range(cfg.L) if l % 3 != 1]
    K[:, marked, :, t, 0] = 250.0 * np.sqrt(d)   # logit 8 * 250 = 2000
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    assert skv.shotkv_repaired_items(ctx) == cfg.B * len(marked) * cfg.Hkv
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p)
    ctx.close()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mean", [20, 50, 66])
def test_out_of_range_among_short_units(mean, d):
    """Units on both sides of the length below which a piece's sum is not looked at for itself: the item of the one
    key out of range is recomputed and no other."""
    ctx = skv.Context(0)
    S = 1800 // mean
    cfg = wl.PrefillConfig("short", B=1, L=4, H=32, Hkv=8, d=d, N=S * mean + 150, W=64, S=S, shot_dist="uniform", shot_lo=mean - 6,
                           shot_hi=mean + 6, question_len=150, r_p=0.5, cfg_id=27)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    Q[..., 0], K[..., 0] = 8.0, 0.0
    t = 7 * 128 + 41
    K[0, 2, :, t, 0] = 250.0 * np.sqrt(d)        # logit 8 * 250 = 2000
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    assert skv.shotkv_repaired_items(ctx) == cfg.Hkv
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p, check_tokens=False)
    ctx.close()


@pytest.mark.parametrize("d,G,W", [(64, 3, 33), (128, 3, 33), (128, 5, 45), (64, 7, 9)], ids=["99_rows", "99_rows_d128", "225_rows", "63_rows"])
def test_token_importance_of_wide_logits(d, G, W):
    """Logits of a standard deviation of 400 beside rows that fill the operand up (the next unit's queries, so their logits are as
    wide): those carry no weight.  In units of log2 a logit stays below 4,000, where fp32 resolves 2.4e-4; a few such
    roundings in the dot product and in its reference make 1e-3 of a weight."""
    ctx = skv.Context(0)
    L, Hkv, N = 2, 2, 3000
    g = torch.Generator(device="cuda").manual_seed(1)
    Q = (20 * torch.randn(1, L, G * Hkv, W, d, generator=g, device="cuda")).bfloat16()
    K = (20 * torch.randn(1, L, Hkv, N, d, generator=g, device="cuda")).bfloat16()
    dims = skv.make_dims(1, L, G * Hkv, Hkv, d, N, W, 0)
    imp = torch.zeros(1, L, Hkv, N, device="cuda")
    ws = torch.empty(skv.shotkv_workspace_bytes(dims), dtype=torch.uint8, device="cuda")
    skv.shotkv_prefill_score(ctx, dims, Q, K, imp, ws)
    x = torch.einsum("blhgwd,blhnd->blhgwn", Q.double().view(1, L, Hkv, G, W, d), K.double()) / d ** 0.5
    own = N - W + torch.arange(W, device="cuda")
    want = x.masked_fill_(torch.arange(N, device="cuda") > own[:, None], float("-inf")).softmax(-1).sum((3, 4))
    assert torch.isfinite(imp).all()
    assert (imp.double() - want).norm() <= 1e-3 * want.norm()
    ctx.close()
