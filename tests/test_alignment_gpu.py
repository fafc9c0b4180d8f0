"""bf16 tensors that do not begin on a 16-byte boundary (a contiguous view at an odd offset) are refused on the
host: the kernels read them as 16-byte vectors.  Nothing of a refused call is enqueued."""
import pytest
import torch

import paper_2502_01941_b200 as skv

pytestmark = pytest.mark.gpu

B, L, H, Hkv, d, N, W, S = 1, 2, 8, 2, 64, 300, 8, 3


@pytest.fixture(scope="module")
def ctx():
    c = skv.Context(0)
    yield c
    c.close()


def _off(t):
    """The same tensor 2 bytes behind a 16-byte boundary."""
    flat = torch.zeros(t.numel() + 8, dtype=t.dtype, device=t.device)
    v = flat[1:1 + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.is_contiguous() and v.data_ptr() % 16 == 2
    return v


def _refused(call):
    with pytest.raises(skv.ShotKVError, match="16-byte aligned"):
        call()


@pytest.mark.parametrize("flags", [0, skv.FLAG_TOKEN_IMPORTANCE])
@pytest.mark.parametrize("which", ["Q", "K", "V", "Kc", "Vc"])
def test_prefill(ctx, which, flags):
    dims, pol = skv.make_dims(B, L, H, Hkv, d, N, W, S), skv.make_policy(r_p=0.5)
    off = torch.tensor([[10, 90, 150, 250]], dtype=torch.int32).numpy()
    m = skv.shotkv_kept_capacity(dims, pol, off)
    o = skv.alloc_prefill_outputs(dims, m, token_importance=True)
    t = dict(Q=torch.randn(B, L, H, W, d, device="cuda").bfloat16(), K=torch.randn(B, L, Hkv, N, d, device="cuda").bfloat16(),
             V=torch.randn(B, L, Hkv, N, d, device="cuda").bfloat16(), Kc=o["Kc"], Vc=o["Vc"])
    t[which] = _off(t[which])
    _refused(lambda: skv.shotkv_prefill_compress(ctx, dims, pol, t["Q"], t["K"], t["V"], off, o["shot_scores"], o["keep"], o["kept_idx"],
                                                 o["kept_count"], m, t["Kc"], t["Vc"], o["token_importance"], flags, o["ws"]))
    if which != "Q":
        _refused(lambda: skv.shotkv_compact_kv(ctx, dims, t["K"], t["V"], o["kept_idx"], o["kept_count"], m, t["Kc"], t["Vc"]))
    torch.cuda.synchronize()


@pytest.mark.parametrize("which", ["Kd", "Vd", "q", "k", "v", "Kc", "Vc"])
def test_decode(ctx, which):
    M, cap = 40, 8
    dims, pol = skv.make_dims(B, L, H, Hkv, d, 1, 1, 0), skv.make_policy(r_d=0.5, recompress_every=4)

    def bf(*shape):
        return torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")

    t = dict(Kd=bf(B, L, Hkv, cap, d), Vd=bf(B, L, Hkv, cap, d), q=bf(B, L, H, d), k=bf(B, L, Hkv, d), v=bf(B, L, Hkv, d),
             Kc=bf(B, L, Hkv, M, d), Vc=bf(B, L, Hkv, M, d))
    t[which] = _off(t[which])
    acc, born = torch.zeros(B, L, cap, device="cuda"), torch.zeros(B, L, cap, dtype=torch.int32, device="cuda")
    ws = torch.empty(skv.shotkv_decode_workspace_bytes(dims, cap), dtype=torch.uint8, device="cuda")
    kept = torch.full((B, L), M, dtype=torch.int32, device="cuda")
    out = torch.zeros(B, L, H, d, device="cuda")
    init = lambda: skv.shotkv_decode_init(ctx, dims, pol, cap, M, t["Kd"], t["Vd"], acc, born, ws)
    if which in ("Kd", "Vd"):
        return _refused(init)
    st = init()
    _refused(lambda: skv.shotkv_decode_step_attend(ctx, st, t["q"], t["k"], t["v"], t["Kc"], t["Vc"], kept, out))
    if which != "Vc":
        _refused(lambda: skv.shotkv_decode_step(ctx, st, t["q"], t["k"], t["v"], t["Kc"], kept))
    assert st.T == 0 and st.n_dec == 0
    torch.cuda.synchronize()
