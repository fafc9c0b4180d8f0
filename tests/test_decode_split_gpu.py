"""Units shared by a cluster of CTAs and the fused end of an eviction cycle, against the oracle: one to
sixteen CTAs to a unit, CTAs without a single key, heads that do not divide by the cluster, regions on
both sides of the ranking by counting (256 entries) and by sorting."""
import numpy as np
import pytest
import torch

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import workloads as wl
import parity as P
from test_decode_gpu import GpuDecoder, OUT_ATOL, OUT_RTOL, lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = skv.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("attend", [False, True], ids=["plain", "attend"])
@pytest.mark.parametrize("Hkv,G,d,M,count", [(1, 4, 128, 2048, 2048), (1, 8, 64, 2047, 1), (2, 3, 128, 2049, 0), (2, 4, 64, 500, 400),
                                             (8, 4, 128, 1100, 1023), (9, 1, 64, 700, 513), (96, 1, 64, 1500, 1400)])
def test_unit_shared_by_a_cluster(ctx, Hkv, G, d, M, count, attend):
    cfg = wl.DecodeConfig("split", B=1, L=1, H=Hkv * G, Hkv=Hkv, d=d, steps=14, r_d=0.5, recompress_every=4, cfg_id=71)
    assert lockstep(ctx, cfg, M, [(0, 0)], np.full((1, 1), count, np.int32), attend=attend) <= 1


@pytest.mark.parametrize("Hkv,G,d,M,count", [(1, 1, 64, 4096, 4000), (1, 7, 128, 4100, 4100), (1, 5, 64, 3000, 2999), (2, 8, 128, 5000, 4999),
                                             (3, 3, 128, 3000, 2990), (7, 2, 64, 6000, 5900)])
def test_unit_shared_by_more_than_eight(ctx, Hkv, G, d, M, count):
    """Clusters of nine to sixteen, output elements that do and do not divide by them, for both steps."""
    cfg = wl.DecodeConfig("split", B=1, L=1, H=Hkv * G, Hkv=Hkv, d=d, steps=6, r_d=0.5, recompress_every=4, cfg_id=76)
    for attend in (False, True):
        assert lockstep(ctx, cfg, M, [(0, 0)], np.full((1, 1), count, np.int32), attend=attend) <= 1


@pytest.mark.parametrize("every", [255, 256, 257, 300, 530])
def test_eviction_of_a_large_region(ctx, every):
    cfg = wl.DecodeConfig("evict", B=1, L=1, H=4, Hkv=2, d=64, steps=every + 3, r_d=0.6, recompress_every=every, cfg_id=72)
    assert lockstep(ctx, cfg, 40, [(0, 0)]) <= 2


@pytest.mark.parametrize("attend", [False, True], ids=["plain", "attend"])
@pytest.mark.parametrize("Hkv,G,d,M,every,steps,one", [
    (1, 8, 128, 3000, 1, 6, (3, 3)),            # nine and sixteen CTAs to the unit: no eviction in the first kernel, every second step
    (1, 8, 128, 2000, 1, 6, (6, 3)),            # six and sixteen
    (1, 8, 128, 600, 1, 6, (0, 6)),             # one, which is no cluster, and seven
    (2, 4, 64, 30, 1, 6, (6, 6)), (5, 3, 128, 64, 3, 8, (8, 8)), (8, 2, 128, 100, 4, 9, (9, 9)),
    (16, 1, 64, 30, 2, 6, (3, 3)), (17, 1, 64, 30, 2, 6, (0, 0)),                          # heads
    (2, 2, 64, 20, 127, 130, (130, 130)), (2, 2, 64, 20, 128, 131, (131, 131)),            # entries when it evicts
    (2, 2, 128, 20, 129, 132, (132, 131)), (16, 1, 64, 20, 400, 259, (256, 150))])         # weights; from 171 keys on two CTAs a unit
def test_step_of_one_cluster(ctx, Hkv, G, d, M, every, steps, one, attend):
    """A (sequence, layer) whose CTAs are one cluster ends its step in the first kernel: `one` of the steps do, scores only and
    with the attention output, on both sides of where that stops: 16 CTAs (8 when it evicts), 4,096 weights, evictions of 128
    entries (with the attention output)."""
    cfg = wl.DecodeConfig("one", B=2, L=1, H=Hkv * G, Hkv=Hkv, d=d, steps=steps, r_d=0.5, recompress_every=every, cfg_id=77)
    before = skv.shotkv_launch_count(ctx)
    assert lockstep(ctx, cfg, M, [(0, 0), (1, 0)], np.array([[M], [M - 7]], np.int32), attend=attend) <= 2
    assert skv.shotkv_launch_count(ctx) - before == 2 * steps - one[attend]


@pytest.mark.parametrize("M", [40, 2048], ids=["whole_unit", "shared_unit"])
def test_query_that_is_not_a_number_gives_no_output(ctx, M):
    """The same output, zero, whether one CTA has the unit or a cluster shares it; other heads are as without it."""
    cfg = wl.DecodeConfig("nan", B=1, L=1, H=8, Hkv=2, d=128, steps=4, r_d=0.5, recompress_every=4, cfg_id=74)
    Kc, kept = wl.random_prefill_cache(cfg, M, "cuda")
    Vc = wl.random_prefill_values(cfg, M, "cuda")
    gpu = GpuDecoder(ctx, cfg, Kc, kept, Vc=Vc)
    q, k, v = wl.decode_step_inputs(cfg, 0, "cuda")
    q[0, 0, 2] = float("nan")
    gpu.step(q, k, v)
    torch.cuda.synchronize()
    n = int(kept[0, 0])
    keys = torch.cat([Kc[0, 0, :, :n], k[0, 0][:, None]], 1).double().repeat_interleave(4, 0)
    vals = torch.cat([Vc[0, 0, :, :n], v[0, 0][:, None]], 1).double().repeat_interleave(4, 0)
    want = ((q[0, 0].double()[:, None] * keys).sum(-1) / 128 ** 0.5).softmax(-1)[:, None] @ vals
    want[2] = 0
    err = (gpu.out[0, 0].double() - want[:, 0]).abs()
    assert (err <= OUT_RTOL * want[:, 0].abs().amax(1, keepdim=True) + OUT_ATOL).all(), err.amax(1)


@pytest.mark.parametrize("L", [19, 32, 37, 55, 56, 74, 75])
def test_whole_units_two_to_an_sm(ctx, L):
    """More units than SMs and at most two to an SM, and three to four times as many, an eviction among the steps."""
    cfg = wl.DecodeConfig("pairs", B=1, L=L, H=32, Hkv=8, d=128, steps=9, r_d=0.5, recompress_every=4, cfg_id=75)
    assert lockstep(ctx, cfg, 300, [(0, 0), (0, L - 1)], attend=True) <= 1


@pytest.mark.parametrize("L,Hkv,G,d,M,Dcap", [(1, 1, 8, 128, 6000, 4096), (1, 2, 8, 128, 3000, 1500), (2, 8, 4, 128, 3276, 750), (1, 16, 1, 64, 60, 4096),
                                              (1, 16, 8, 128, 40, 2100)])
def test_clusters_of_ctas_that_take_much_memory(ctx, L, Hkv, G, d, M, Dcap):
    """Decode regions of which two or one fit an SM: units shared by up to sixteen CTAs, and steps of sixteen heads that end in
    their first kernel."""
    cfg = wl.DecodeConfig("room", B=1, L=L, H=Hkv * G, Hkv=Hkv, d=d, steps=2 * (Dcap - 4), r_d=0.5, recompress_every=4, cfg_id=79)
    assert cfg.Dcap == Dcap
    for attend in (False, True):
        assert lockstep(ctx, cfg, M, [(0, 0)], np.full((1, L), M, np.int32), steps=5, attend=attend) <= 1


@pytest.mark.parametrize("d,L", [(128, 55), (128, 56), (128, 74), (128, 75), (64, 28), (64, 32), (64, 37), (64, 92), (64, 93), (64, 127)])
def test_whole_units_on_both_sides_of_a_wave(ctx, d, L):
    """Units that are scored two and four blocks of keys deep, shared and whole, one wave of them and more."""
    cfg = wl.DecodeConfig("waves", B=1, L=L, H=16, Hkv=8, d=d, steps=5, r_d=0.5, recompress_every=4, cfg_id=80)
    assert lockstep(ctx, cfg, 1400, [(0, 0), (0, L - 1)], np.full((1, L), 1311, np.int32)) <= 1


def test_entries_of_whole_units(ctx):
    """The attention-output step of units that no cluster shares, with more decode entries than a CTA has threads."""
    cfg = wl.DecodeConfig("entries", B=1, L=20, H=24, Hkv=8, d=64, steps=133, r_d=0.5, recompress_every=131, cfg_id=81)
    assert lockstep(ctx, cfg, 30, [(0, 7)], np.full((1, 20), 29, np.int32), attend=True) <= 1


@pytest.mark.parametrize("G,d", [(1, 64), (3, 128), (5, 64), (8, 128)])
@pytest.mark.parametrize("attend,most", [(False, 1024), (True, 400)], ids=["plain", "attend"])
def test_many_entries(ctx, G, d, attend, most):
    """Steps on both sides of the number of entries up to which they end in their first kernel, rows in two halves of four."""
    cfg = wl.DecodeConfig("many", B=1, L=1, H=2 * G, Hkv=2, d=d, steps=most + 3, r_d=0.9, recompress_every=most + 3, cfg_id=82)
    Kc, kept = wl.random_prefill_cache(cfg, 40, "cuda", np.full((1, 1), 37, np.int32))
    gpu = GpuDecoder(ctx, cfg, Kc, kept, Vc=wl.random_prefill_values(cfg, 40, "cuda") if attend else None)
    g = torch.Generator(device="cuda").manual_seed(5)
    n = most - 2
    for x in (gpu.Kd, gpu.Vd):
        x.copy_(torch.randn(x.shape, generator=g, device="cuda"))
    gpu.acc.copy_(torch.rand(gpu.acc.shape, generator=g, device="cuda"))
    gpu.state.T = gpu.state.n_dec = n
    for one in (True, True, False, False):
        q, k, v = wl.decode_step_inputs(cfg, n, "cuda")
        want = gpu.acc[0, 0, :n].double()
        before = skv.shotkv_launch_count(ctx)
        gpu.step(q, k, v)
        torch.cuda.synchronize()
        assert skv.shotkv_launch_count(ctx) - before == (1 if one else 2)
        n += 1
        keys = torch.cat([Kc[0, 0, :, :37], gpu.Kd[0, 0, :, :n]], 1).double()
        w = ((q[0, 0].double().view(2, G, 1, d) * keys[:, None]).sum(-1) / d ** 0.5).softmax(-1)
        want = torch.cat([want, want.new_zeros(1)]) + w[:, :, 37:].sum((0, 1))
        np.testing.assert_allclose(gpu.acc[0, 0, :n].double().cpu().numpy(), want.cpu().numpy(), rtol=P.SCORE_RTOL, atol=P.SCORE_ATOL)
