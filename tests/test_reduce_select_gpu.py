"""The kernel that reduces the scoring pass's partials and selects, and the ranking shared with
shotkv_select_shots: sizes on both sides of every branch (ranking by counting or by sorting, shots
to a warp, kv heads to a cluster)."""
import numpy as np
import pytest
import torch

import paper_2502_01941_b200 as skv
from oracle import shotkv_oracle as O
from paper_2502_01941_b200 import workloads as wl
import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = skv.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("S", [1, 2, 31, 33, 255, 256, 257, 511, 512, 513, 1025, 8192])
def test_ranking_with_ties(ctx, S):
    """Whole numbers, so that many scores tie (index order decides), zeros of both signs among them."""
    B, L, W = 2, 2, 4
    rng = np.random.default_rng(S)
    off = np.concatenate([np.zeros((B, 1), np.int64) + 3, 3 + np.cumsum(rng.integers(1, 9, size=(B, S)), axis=1)], axis=1).astype(np.int32)
    N = int(off[:, -1].max()) + 20
    dims = skv.make_dims(B, L, 4, 2, 64, N, W, S)
    sc = rng.integers(-3, 4, size=(B, L, S)).astype(np.float32)
    sc[sc == 0] = np.where(rng.random((sc == 0).sum()) < 0.5, np.float32(-0.0), np.float32(0.0))
    for mode in (0, 1):
        pol = skv.make_policy(r_p=0.45, select_mode=mode)
        Mcap = skv.shotkv_kept_capacity(dims, pol, off)
        out = skv.alloc_prefill_outputs(dims, Mcap)
        out["shot_scores"].copy_(torch.from_numpy(sc))
        skv.shotkv_select_shots(ctx, dims, pol, None, off, out["shot_scores"], out["keep"], out["kept_idx"], out["kept_count"], Mcap,
                                out["ws"])
        torch.cuda.synchronize()
        for b in range(B):
            for l in range(L):
                keep, idx, _ = O.select_shots(sc[b, l], off[b], N, 0.45, mode)
                np.testing.assert_array_equal(out["keep"][b, l].cpu().numpy(), keep)
                n = int(out["kept_count"][b, l])
                assert n == len(idx)
                np.testing.assert_array_equal(out["kept_idx"][b, l, :n].cpu().numpy(), idx)
                assert (out["kept_idx"][b, l, n:] == -1).all()


@pytest.mark.parametrize("Hkv,G,W", [(1, 4, 32), (3, 2, 16), (8, 4, 64), (9, 1, 8), (17, 3, 64)])
@pytest.mark.parametrize("mode", [skv.SCORING_FAST, skv.SCORING_EXACT], ids=["fast", "exact"])
def test_heads_to_a_cluster(ctx, Hkv, G, W, mode):
    cfg = wl.PrefillConfig("heads", B=2, L=1, H=Hkv * G, Hkv=Hkv, d=64, N=2305, W=W, S=17, shot_dist="uniform", shot_lo=64,
                           shot_hi=192, question_len=129, r_p=0.4, cfg_id=62)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    skv.shotkv_set_scoring_mode(ctx, mode)
    try:
        gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    finally:
        skv.shotkv_set_scoring_mode(ctx, skv.SCORING_FAST)
    assert P.check_all_units(gpu, Q, K, V, off, cfg.r_p) <= 1


@pytest.mark.parametrize("W", [32, 64])                    # 128 and 256 window rows
@pytest.mark.parametrize("mode", [skv.SCORING_FAST, skv.SCORING_EXACT], ids=["fast", "exact"])
@pytest.mark.parametrize("what", ["query_nan", "query_inf", "key_nan"])
def test_rows_that_are_not_numbers_carry_no_weight(ctx, what, mode, W):
    """A window row whose softmax denominator is not a number drops out of the sums; the other rows, and the
    other heads, give what they give without it."""
    Hkv, G, d, N, S = 2, 4, 64, 1500, 7
    cfg = wl.PrefillConfig("nan", B=1, L=1, H=Hkv * G, Hkv=Hkv, d=d, N=N, W=W, S=S, shot_dist="uniform", shot_lo=100, shot_hi=250,
                           question_len=130, r_p=0.4, cfg_id=64)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    dropped = torch.zeros(Hkv * G, W, dtype=torch.bool, device="cuda")
    if what == "key_nan":
        K[0, 0, 1, 296:304, 5] = float("nan")              # every window row sees them (the fast kernels' FMA pipe takes a
                                                           # lone one for a key without weight, the other pipe does not)
        dropped[G:] = True
    else:
        Q[0, 0, 2, 3] = float("nan") if what == "query_nan" else float("inf")
        dropped[2, 3] = True
    x = torch.einsum("hwd,hnd->hwn", Q[0, 0].double(), K[0, 0].double().repeat_interleave(G, 0)) / d ** 0.5
    x = x.masked_fill(torch.arange(N, device="cuda") > torch.arange(N - W, N, device="cuda")[:, None], float("-inf"))
    alpha = torch.where(dropped[..., None], 0.0, x.softmax(-1)).sum((0, 1))
    o = off[0]
    want = torch.stack([alpha[o[i]:o[i + 1]].mean() for i in range(S)])
    skv.shotkv_set_scoring_mode(ctx, mode)
    try:
        got = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")["shot_scores"][0, 0]
    finally:
        skv.shotkv_set_scoring_mode(ctx, skv.SCORING_FAST)
    assert torch.allclose(got.double(), want, rtol=P.SCORE_RTOL, atol=P.SCORE_ATOL), (got, want)


@pytest.mark.parametrize("B,L,S,mean,Hkv", [(1, 1, 3, 200, 1), (1, 297, 1, 130, 1), (2, 40, 7, 97, 2), (1, 37, 65, 129, 8), (1, 2, 40, 33, 3),
                                            (3, 200, 8, 300, 8), (1, 600, 4, 160, 9)])
def test_scores_from_token_importances(ctx, B, L, S, mean, Hkv):
    """Short units, few long ones and many long ones, on both sides of the lines between the kernel's forms, lengths
    around a run of 32 tokens among them.  Two orders of up to 4,000 positive fp32 terms: 1e-5 relative."""
    rng = np.random.default_rng(S)
    lens = np.maximum(1, rng.integers(mean // 2, 3 * mean // 2, size=(B, S)) // 32 * 32 + rng.integers(-1, 2, size=(B, S)))
    off = np.concatenate([np.full((B, 1), 5), 5 + np.cumsum(lens, 1)], 1).astype(np.int32)
    N = int(off.max()) + 40
    dims, pol = skv.make_dims(B, L, Hkv, Hkv, 64, N, 8, S), skv.make_policy(r_p=0.5)
    Mcap = skv.shotkv_kept_capacity(dims, pol, off)
    out = skv.alloc_prefill_outputs(dims, Mcap)
    imp = torch.rand(B, L, Hkv, N, device="cuda", generator=torch.Generator("cuda").manual_seed(S))
    skv.shotkv_select_shots(ctx, dims, pol, imp, off, out["shot_scores"], out["keep"], out["kept_idx"], out["kept_count"], Mcap, out["ws"])
    total = torch.nn.functional.pad(imp.double().sum(2).cumsum(-1), (1, 0))
    for b in range(B):
        o = torch.from_numpy(off[b]).long().cuda()
        want = (total[b][:, o[1:]] - total[b][:, o[:-1]]) / (o[1:] - o[:-1])
        assert torch.allclose(out["shot_scores"][b].double(), want, rtol=1e-5, atol=0)


@pytest.mark.parametrize("S,L", [(1440, 1), (1475, 1), (1475, 2)])
def test_clusters_of_ctas_that_fill_an_sm(ctx, S, L):
    """256 window rows, more shots than leave two CTAs of the reduction room on an SM."""
    cfg = wl.PrefillConfig("many", B=1, L=L, H=32, Hkv=8, d=64, N=23680, W=64, S=S, shot_dist="uniform", shot_lo=10,
                           shot_hi=24, question_len=200, r_p=0.3, cfg_id=63)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p, units=[(0, L - 1)], check_tokens=False)


@pytest.mark.parametrize("L", [27, 28])
def test_more_clusters_than_one_wave(ctx, L):
    """256 window rows on both sides of three CTAs to an SM (444): four and three pieces in flight a warp."""
    cfg = wl.PrefillConfig("waves", B=2, L=L, H=32, Hkv=8, d=64, N=1700, W=64, S=61, shot_dist="uniform", shot_lo=17,
                           shot_hi=31, question_len=150, r_p=0.4, cfg_id=64)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, 0, "fused")
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p, units=[(0, 0), (0, L - 1), (1, L - 1)], check_tokens=False)
