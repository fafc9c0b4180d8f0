"""The calls of a program's inner loops by both ways of marshalling their arguments: the same results, and
the same exception for an argument that is not what the call takes."""
import numpy as np
import pytest
import torch

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import binding, workloads as wl
import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(params=["module", "ctypes"])
def ctx(request, monkeypatch):
    c = skv.Context(0)
    assert binding._native is not None
    if request.param == "ctypes":
        monkeypatch.setattr(binding, "_native", None)
    yield c
    c.close()


def _case():
    cfg = wl.PrefillConfig("marshal", B=2, L=2, H=8, Hkv=2, d=64, N=700, W=16, S=5, shot_dist="uniform", shot_lo=60,
                           shot_hi=200, question_len=50, r_p=0.4, cfg_id=26)
    return cfg, wl.prefill_batch(cfg, "cuda")


@pytest.mark.parametrize("path", ["fused", "fused_tokens", "calls"])
@pytest.mark.parametrize("offsets", ["int32", "int64", "strided", "tensor", "longer"])
def test_prefill_calls(ctx, path, offsets):
    cfg, (Q, K, V, off) = _case()
    o = {"int32": off, "int64": off.astype(np.int64), "strided": np.repeat(off, 2, axis=1)[:, ::2], "tensor": torch.from_numpy(off),
         "longer": np.concatenate([off, off])}[offsets]
    gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, o, cfg.r_p, 0, path)
    P.check_all_units(gpu, Q, K, V, off, cfg.r_p)


@pytest.mark.parametrize("what,error", [("dtype", TypeError), ("host", ValueError), ("strided", ValueError), ("list", TypeError)])
def test_arguments_that_are_refused(ctx, what, error):
    cfg, (Q, K, V, off) = _case()
    dims, pol = P.dims_of(cfg), skv.make_policy(r_p=cfg.r_p)
    bad = {"dtype": Q.float(), "host": Q.cpu(), "strided": Q.transpose(-1, -2).contiguous().transpose(-1, -2), "list": [1.0]}[what]
    mcap = skv.shotkv_kept_capacity(dims, pol, off)
    o = skv.alloc_prefill_outputs(dims, mcap, token_importance=True)
    with pytest.raises(error, match="Qwin"):
        skv.shotkv_prefill_score(ctx, dims, bad, K, o["token_importance"], o["ws"])
    with pytest.raises(error, match="Qwin"):
        skv.shotkv_prefill_compress(ctx, dims, pol, bad, K, V, off, o["shot_scores"], o["keep"], o["kept_idx"], o["kept_count"], mcap,
                                    o["Kc"], o["Vc"], None, 0, o["ws"])
    with pytest.raises(skv.ShotKVError):                     # the library's own checks, through either way
        skv.shotkv_prefill_compress(ctx, dims, pol, Q, K, V, off, o["shot_scores"], o["keep"], o["kept_idx"], o["kept_count"], 1,
                                    o["Kc"], o["Vc"], None, 0, o["ws"])


@pytest.mark.parametrize("attend", [False, True])
def test_decode_steps_on_another_stream(ctx, attend):
    """The current stream is the one a call goes to; a stream given as an argument goes before it."""
    B, L, H, Hkv, d, M, steps = 2, 2, 8, 2, 64, 90, 6
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()
    dims, pol = skv.make_dims(B, L, H, Hkv, d, M + 8, 8, 1), skv.make_policy(r_d=0.5, recompress_every=4)
    cap = skv.shotkv_decode_capacity(pol, steps)
    Kc, Vc = rnd(B, L, Hkv, M, d), rnd(B, L, Hkv, M, d)
    kept = torch.full((B, L), M, dtype=torch.int32, device="cuda")
    ins = [(rnd(B, L, H, d), rnd(B, L, Hkv, d), rnd(B, L, Hkv, d)) for _ in range(steps)]
    torch.cuda.synchronize()
    results = []
    for how in ("default", "current", "argument"):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s if how == "current" else torch.cuda.default_stream()):
            Kd = torch.zeros(B, L, Hkv, cap, d, dtype=torch.bfloat16, device="cuda")
            Vd, out = torch.zeros_like(Kd), torch.zeros(B, L, H, d, device="cuda")
            acc, born = torch.zeros(B, L, cap, device="cuda"), torch.zeros(B, L, cap, dtype=torch.int32, device="cuda")
            ws = torch.zeros(skv.shotkv_decode_workspace_bytes(dims, cap), dtype=torch.uint8, device="cuda")
            st = skv.shotkv_decode_init(ctx, dims, pol, cap, M, Kd, Vd, acc, born, ws)
            s.wait_stream(torch.cuda.default_stream())
            arg = s if how == "argument" else None
            for q, k, v in ins:
                if attend:
                    skv.shotkv_decode_step_attend(ctx, st, q, k, v, Kc, Vc, kept, out, stream=arg)
                else:
                    skv.shotkv_decode_step(ctx, st, q, k, v, Kc, kept, stream=arg)
            torch.cuda.synchronize()
            n = st.n_dec
            results.append([t.cpu() for t in (acc[:, :, :n], born[:, :, :n], Kd[:, :, :, :n], out)])
    for r in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, results[0]))
    assert float(results[0][0].sum()) > 0
