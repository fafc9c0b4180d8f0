"""Kernels are launched so that they may begin before the one ahead of them on the stream has ended;
what precedes and follows a call on its stream must not notice: inputs that arrive by a copy, by a
slow kernel or from another stream, and buffers that are overwritten right behind a call."""
import pytest
import torch

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import workloads as wl
import parity as P

pytestmark = pytest.mark.gpu

SLEEP = 3_000_000          # cycles: some milliseconds, far longer than the calls below


@pytest.fixture(scope="module")
def ctx():
    c = skv.Context(0)
    yield c
    c.close()


def _outputs(cfg, dims, Mcap):
    return skv.alloc_prefill_outputs(dims, Mcap, token_importance=True)


@pytest.mark.parametrize("how", ["copy", "kernel", "other_stream"])
@pytest.mark.parametrize("path", ["fused", "tokens"])
@pytest.mark.parametrize("W", [32, 64])
def test_prefill_between_other_work(ctx, how, path, W):
    cfg = wl.CONFIGS[2].replace(name="order", B=1, L=2, N=3001, S=9, W=W, shot_lo=20, shot_hi=900, question_len=150)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    dims, pol = P.dims_of(cfg), skv.make_policy(r_p=0.3)
    Mcap = skv.shotkv_kept_capacity(dims, pol, off)
    flags = skv.FLAG_TOKEN_IMPORTANCE if path == "tokens" else 0

    def call(K_, V_, o):
        skv.shotkv_prefill_compress(ctx, dims, pol, Q, K_, V_, off, o["shot_scores"], o["keep"], o["kept_idx"], o["kept_count"],
                                    Mcap, o["Kc"], o["Vc"], o["token_importance"], flags, o["ws"])

    ref = _outputs(cfg, dims, Mcap)
    call(K, V, ref)
    torch.cuda.synchronize()
    hostK, hostV = K.cpu().pin_memory(), V.cpu().pin_memory()
    Kin, Vin, out = torch.zeros_like(K), torch.zeros_like(V), _outputs(cfg, dims, Mcap)
    side = torch.cuda.Stream()
    for _ in range(5):
        Kin.zero_(); Vin.zero_()
        for n in ("shot_scores", "keep", "kept_idx", "kept_count", "Kc", "Vc", "token_importance"):
            out[n].zero_()
        if how == "copy":
            torch.cuda._sleep(SLEEP)
            Kin.copy_(hostK, non_blocking=True); Vin.copy_(hostV, non_blocking=True)
        elif how == "kernel":
            torch.cuda._sleep(SLEEP)
            torch.add(K, 0, out=Kin); torch.add(V, 0, out=Vin)
        else:
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                torch.cuda._sleep(SLEEP)
                Kin.copy_(K); Vin.copy_(V)
            torch.cuda.current_stream().wait_stream(side)
        call(Kin, Vin, out)
        Kin.zero_(); Vin.zero_()                       # right behind the call
        kept = out["Kc"].clone()
        torch.cuda.synchronize()
        for n in ("shot_scores", "keep", "kept_idx", "kept_count"):
            assert torch.equal(out[n], ref[n]), n
        assert torch.equal(kept, ref["Kc"]) and torch.equal(out["Vc"], ref["Vc"])
        if flags:
            assert torch.equal(out["token_importance"], ref["token_importance"])


def test_decode_between_other_work(ctx):
    cfg = wl.DecodeConfig("order", B=1, L=2, H=8, Hkv=2, d=128, steps=12, r_d=0.5, recompress_every=3, cfg_id=73)
    Kc, kept = wl.random_prefill_cache(cfg, 700, "cuda")
    Vc = wl.random_prefill_values(cfg, 700, "cuda")
    dims, pol = skv.make_dims(1, 2, 8, 2, 128, 1, 1, 0), skv.make_policy(r_d=0.5, recompress_every=3)
    Dcap = skv.shotkv_decode_capacity(pol, 12)

    def run(slow):
        Kd = torch.zeros(1, 2, 2, Dcap, 128, dtype=torch.bfloat16, device="cuda")
        Vd, acc = torch.zeros_like(Kd), torch.zeros(1, 2, Dcap, device="cuda")
        born = torch.zeros(1, 2, Dcap, dtype=torch.int32, device="cuda")
        ws = torch.empty(skv.shotkv_decode_workspace_bytes(dims, Dcap), dtype=torch.uint8, device="cuda")
        st = skv.shotkv_decode_init(ctx, dims, pol, Dcap, 700, Kd, Vd, acc, born, ws)
        q, k, v = (torch.zeros_like(t) for t in wl.decode_step_inputs(cfg, 0, "cuda"))
        attn, all_attn = torch.zeros(1, 2, 8, 128, device="cuda"), []
        for s in range(12):
            new = wl.decode_step_inputs(cfg, s, "cuda")
            if slow:
                torch.cuda._sleep(SLEEP // 4)
            for a, b in zip((q, k, v), new):
                torch.add(b, 0, out=a)
            skv.shotkv_decode_step_attend(ctx, st, q, k, v, Kc, Vc, kept, attn)
            q.zero_(); k.zero_(); v.zero_()            # right behind the call
            all_attn.append(attn.clone())
        torch.cuda.synchronize()
        n = st.n_dec
        return acc[:, :, :n], born[:, :, :n], Kd[:, :, :, :n], Vd[:, :, :, :n], torch.stack(all_attn)

    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)
