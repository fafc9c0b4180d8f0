"""What a user of this library has it do, as cases that can be timed.

A case is a dict of plain sizes and options; `prepare` makes what the calling program holds before
the call (seeded inputs on the GPU, output buffers, workspaces, decode states), `run` makes one pass
through the public calls and returns all of their outputs, `work` counts the bytes and operations
the pass cannot do without, `tolerance` says how far two correct implementations may be apart.

Four kinds of pass:
  compress     shotkv_prefill_compress, the whole of the prefill phase in one call
  importance   shotkv_prefill_score, shotkv_select_shots, shotkv_compact_kv: the same phase in three
               calls, for programs that also want the per-token importances
  host         shotkv_prefill_compress_host on page-locked host tensors
  decode       one eviction cycle of the decode phase: `every` steps of shotkv_decode_step (or of
               shotkv_decode_step_attend), the last of which evicts
"""
import functools
import math

import numpy as np
import torch

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import workloads as wl


def _shots(name, kind, B, L, H, Hkv, d, N, W, S, dist, lo, hi, question, preamble=0, r_p=0.2, mode=0):
    return dict(name=name, kind=kind, B=B, L=L, H=H, Hkv=Hkv, d=d, N=N, W=W, S=S, dist=dist, lo=lo, hi=hi,
                question=question, preamble=preamble, r_p=r_p, mode=mode)


def _decode(name, B, L, H, Hkv, d, M, steps, every, r_d, attend):
    return dict(name=name, kind="decode", B=B, L=L, H=H, Hkv=Hkv, d=d, M=M, steps=steps, every=every, r_d=r_d,
                attend=attend)


def listed():
    return [
        # the smallest prefill: one layer of a small model on a 512-token prompt; latency and launches
        _shots("compress_tiny", "compress", 1, 1, 4, 2, 64, 512, 16, 8, "uniform", 40, 70, -1, r_p=0.4),
        # one layer of a 4K few-shot prompt: a program that compresses each layer as its prefill ends
        _shots("compress_layer_4k", "compress", 1, 1, 32, 8, 128, 4096, 32, 16, "uniform", 150, 300, 200),
        # all layers of a 16K prompt at once, shots of very different lengths
        _shots("compress_model_16k", "compress", 1, 32, 32, 8, 128, 16384, 32, 48, "lognormal", 40, 1600, 300),
        # the largest: a batch of four 32K prompts, wide window (256 rows a KV head), small budget
        _shots("compress_batch_32k", "compress", 4, 32, 32, 8, 128, 32768, 64, 96, "uniform", 200, 480, 500, r_p=0.1),
        # nothing a round number: three query heads to a KV head, odd prompt, window and preamble,
        # shots that do not fit are skipped
        _shots("compress_ragged", "compress", 3, 4, 24, 8, 128, 5003, 33, 13, "uniform", 150, 700, 171, preamble=37,
               r_p=0.35, mode=1),
        # sentences as the units that are kept whole
        _shots("compress_sentences_16k", "compress", 1, 32, 32, 8, 128, 16384, 32, 643, "uniform", 10, 40, 300),
        # per-token importances asked for, 256 rows a KV head
        _shots("importance_8k", "importance", 1, 16, 32, 8, 128, 8192, 64, 24, "uniform", 200, 480, 300),
        # tensors in page-locked host memory: an offloaded cache that is compressed on its way back
        _shots("host_8k", "host", 1, 8, 32, 8, 128, 8192, 32, 24, "uniform", 200, 480, 300),
        # generation of eight sequences, scores only: all layers in one call, evicting every 32 steps
        _decode("decode_model_b8", 8, 32, 32, 8, 128, 3276, 512, 32, 0.25, False),
        # the same with the attention output of the step fused in
        _decode("decode_attend_model_b8", 8, 32, 32, 8, 128, 3276, 512, 32, 0.25, True),
        # the fused step as a model calls it: layer after layer, so one layer of a small batch a call
        _decode("decode_attend_layer_b4", 4, 1, 32, 8, 128, 3276, 512, 32, 0.25, True),
        # the smallest decode: one small layer, scores only, evicting at every step
        _decode("decode_tiny", 1, 1, 4, 2, 64, 204, 257, 1, 0.5, False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compress", "compress", "compress", "importance", "host", "decode", "decode", "decode"])
    d = rng.choice([64, 128, 128])
    Hkv = rng.choice([1, 2, 4, 8, 8])
    if kind == "decode":
        G = rng.choice([1, 2, 3, 4, 4, 7, 8])
        B, L, M = _log_int(rng, 1, 8), rng.choice([1, 1, 1, _log_int(rng, 2, 32)]), _log_int(rng, 64, 8192)
        every = rng.choice([1, 8, 32, 32])
        steps = _log_int(rng, 2 * every, 1024)
        # at least one entry goes at the end of the cycle, and no more is read than in the largest listed case
        while B * L * Hkv * (M + 512) * d > 8 * 32 * 8 * 3500 * 128 * 32 // every:
            L = (L + 1) // 2
            M = max(64, M // 2)
        c = _decode("", B, L, G * Hkv, Hkv, d, M, steps, every, round(rng.uniform(0.2, 0.7), 2), rng.random() < 0.6)
    else:
        G = rng.choice([1, 2, 3, 4, 4, 4, 7, 8])
        W = rng.choice([8, 16, 32, 32, 64, rng.randint(5, 70)])
        W = min(W, 256 // G)
        N = _log_int(rng, 512, 32768)
        B, L = _log_int(rng, 1, 4), rng.choice([1, _log_int(rng, 1, 32)])
        most = {"compress": 1 << 30, "importance": 1 << 29, "host": 1 << 27}[kind]     # elements of K
        while B * L * Hkv * N * d > most:
            B, L = (B + 1) // 2, (L + 1) // 2
            if B == L == 1:
                break
        preamble = rng.choice([0, 0, rng.randint(1, N // 20)])
        question = rng.randint(W, max(W, N // 10))
        mean = min(_log_int(rng, 14, 700), (N - preamble - question) // 2)
        S = (N - preamble - question) // mean
        c = _shots("", kind, B, L, G * Hkv, Hkv, d, N, W, S, "uniform", max(1, mean // 2), 2 * mean, question, preamble,
                   round(rng.uniform(0.2, 0.8), 2), rng.choice([0, 1]))
    del c["name"]
    return c


@functools.lru_cache(maxsize=1)
def _context():
    """One context for the process, as a program that serves one GPU keeps."""
    return skv.Context(0)


def _dims(c, N=1, W=1, S=0):
    return skv.make_dims(c["B"], c["L"], c["H"], c["Hkv"], c["d"], c.get("N", N), c.get("W", W), c.get("S", S))


def _prepare_prefill(c, seed):
    cfg = wl.PrefillConfig("case", B=c["B"], L=c["L"], H=c["H"], Hkv=c["Hkv"], d=c["d"], N=c["N"], W=c["W"], S=c["S"],
                           shot_dist=c["dist"], shot_lo=c["lo"], shot_hi=c["hi"], question_len=c["question"],
                           preamble_len=c["preamble"], r_p=c["r_p"], cfg_id=seed)
    dims, policy = _dims(c), skv.make_policy(r_p=c["r_p"], select_mode=c["mode"])
    Q, K, V, offsets = wl.prefill_batch(cfg, "cuda")
    Mcap = skv.shotkv_kept_capacity(dims, policy, offsets)
    if c["kind"] != "host":
        out = skv.alloc_prefill_outputs(dims, Mcap, token_importance=c["kind"] == "importance")
        return dict(kind=c["kind"], ctx=_context(), dims=dims, policy=policy, Q=Q, K=K, V=V, offsets=offsets, Mcap=Mcap, **out)

    def pinned(*shape, dtype):
        return torch.zeros(*shape, dtype=dtype, pin_memory=True)

    B, L, S, Hkv, d = c["B"], c["L"], max(c["S"], 1), c["Hkv"], c["d"]
    host = {n: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for n, t in (("Q", Q), ("K", K), ("V", V))}
    return dict(kind="host", ctx=_context(), dims=dims, policy=policy, offsets=offsets, Mcap=Mcap, **host,
                shot_scores=pinned(B, L, S, dtype=torch.float32), keep=pinned(B, L, S, dtype=torch.uint8),
                kept_idx=pinned(B, L, Mcap, dtype=torch.int32), kept_count=pinned(B, L, dtype=torch.int32),
                Kc=pinned(B, L, Hkv, Mcap, d, dtype=torch.bfloat16), Vc=pinned(B, L, Hkv, Mcap, d, dtype=torch.bfloat16),
                arena=torch.empty(skv.shotkv_host_arena_bytes(dims, Mcap), dtype=torch.uint8, device="cuda"))


def _prepare_decode(c, seed):
    """A generation that has run for `steps - every` steps: the compressed prompt (kept counts differ
    from layer to layer), the entries held after the last eviction with scores that grow with their
    age, and the queries, keys and values of the next `every` steps."""
    cfg = wl.DecodeConfig("case", B=c["B"], L=c["L"], H=c["H"], Hkv=c["Hkv"], d=c["d"], steps=c["steps"], r_d=c["r_d"],
                          recompress_every=c["every"], cfg_id=seed)
    B, L, H, Hkv, d, M, Dcap = cfg.B, cfg.L, cfg.H, cfg.Hkv, cfg.d, c["M"], cfg.Dcap
    T0 = c["steps"] // c["every"] * c["every"] - c["every"]
    n0 = int(cfg.r_d * T0)
    rng = np.random.default_rng(seed)
    counts = rng.integers(M - M // 8, M + 1, size=(B, L)).astype(np.int32)
    Kc, kept_count = wl.random_prefill_cache(cfg, M, "cuda", counts)
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)

    Kd, Vd = normal(B, L, Hkv, Dcap, d), normal(B, L, Hkv, Dcap, d)
    born = torch.zeros(B, L, Dcap, dtype=torch.int32, device="cuda")
    acc = torch.zeros(B, L, Dcap, device="cuda")
    if n0:
        born[:, :, :n0] = torch.rand(B, L, T0, generator=g, device="cuda").argsort(-1)[..., :n0].sort(-1).values
        noise = torch.randn(B, L, n0, generator=g, device="cuda")
        acc[:, :, :n0] = (T0 - born[:, :, :n0]) * (H / (M + n0)) * torch.exp(0.3 * noise)
    dims, policy = _dims(c), skv.make_policy(r_d=c["r_d"], recompress_every=c["every"])
    ws = torch.empty(skv.shotkv_decode_workspace_bytes(dims, Dcap), dtype=torch.uint8, device="cuda")
    ctx = _context()
    s = dict(kind="decode", ctx=ctx, T0=T0, n0=n0, Kc=Kc, kept_count=kept_count, Kd=Kd, Vd=Vd, acc=acc, born=born,
             steps=[wl.decode_step_inputs(cfg, i, "cuda") for i in range(c["every"])],
             st=skv.shotkv_decode_init(ctx, dims, policy, Dcap, M, Kd, Vd, acc, born, ws))
    if c["attend"]:
        s["Vc"] = wl.random_prefill_values(cfg, M, "cuda")
        s["attn"] = torch.zeros(c["every"], B, L, H, d, device="cuda")
        s["attn_steps"] = list(s["attn"])
    return s


def prepare(case, seed):
    return _prepare_decode(case, seed) if case["kind"] == "decode" else _prepare_prefill(case, seed)


def run(s):
    if s["kind"] == "decode":
        st = s["st"]
        st.T, st.n_dec = s["T0"], s["n0"]       # the cycle begins here again
        for i, (q, k, v) in enumerate(s["steps"]):
            if "attn" in s:
                skv.shotkv_decode_step_attend(s["ctx"], st, q, k, v, s["Kc"], s["Vc"], s["kept_count"], s["attn_steps"][i])
            else:
                skv.shotkv_decode_step(s["ctx"], st, q, k, v, s["Kc"], s["kept_count"])
        n = st.n_dec
        out = dict(acc=s["acc"][:, :, :n], born=s["born"][:, :, :n], Kd=s["Kd"][:, :, :, :n], Vd=s["Vd"][:, :, :, :n])
        if "attn" in s:
            out["attn"] = s["attn"]
        return out
    if s["kind"] == "compress":
        skv.shotkv_prefill_compress(s["ctx"], s["dims"], s["policy"], s["Q"], s["K"], s["V"], s["offsets"], s["shot_scores"],
                                    s["keep"], s["kept_idx"], s["kept_count"], s["Mcap"], s["Kc"], s["Vc"], None, 0, s["ws"])
    elif s["kind"] == "host":
        skv.shotkv_prefill_compress_host(s["ctx"], s["dims"], s["policy"], s["Q"], s["K"], s["V"], s["offsets"],
                                         s["shot_scores"], s["keep"], s["kept_idx"], s["kept_count"], s["Mcap"], s["Kc"],
                                         s["Vc"], s["arena"])
    else:
        skv.shotkv_prefill_score(s["ctx"], s["dims"], s["Q"], s["K"], s["token_importance"], s["ws"])
        skv.shotkv_select_shots(s["ctx"], s["dims"], s["policy"], s["token_importance"], s["offsets"], s["shot_scores"],
                                s["keep"], s["kept_idx"], s["kept_count"], s["Mcap"], s["ws"])
        skv.shotkv_compact_kv(s["ctx"], s["dims"], s["K"], s["V"], s["kept_idx"], s["kept_count"], s["Mcap"], s["Kc"], s["Vc"])
    names = ("shot_scores", "keep", "kept_idx", "kept_count", "Kc", "Vc") + (("token_importance",) if s["kind"] == "importance" else ())
    return {n: s[n] for n in names}


def work(case):
    """Every key once, the window queries, the kept rows of K and V read and written; for a decode
    step every cached key (and, with the attention output, every cached value)."""
    c = case
    U, row = c["B"] * c["L"] * c["Hkv"], 2 * c["d"]
    if c["kind"] == "decode":
        T0 = c["steps"] // c["every"] * c["every"] - c["every"]
        keys = c["every"] * (c["M"] - c["M"] // 16 + int(c["r_d"] * T0)) + c["every"] * (c["every"] + 1) // 2
        kept = int(c["r_d"] * (T0 + c["every"]))
        io = c["every"] * c["B"] * c["L"] * c["H"] * c["d"] * (6 if c["attend"] else 2)
        return dict(bytes=U * row * (keys * (2 if c["attend"] else 1) + 4 * c["every"] + 4 * kept // 4) + io,
                    flops=2 * c["B"] * c["L"] * c["H"] * c["d"] * keys * (2 if c["attend"] else 1))
    kept = min(c["N"], max(int(c["r_p"] * c["N"]), c["question"] + c["preamble"]))
    nbytes = U * row * c["N"] + c["B"] * c["L"] * c["H"] * c["W"] * row + U * row * kept * 4 + c["B"] * c["L"] * (kept * 4 + c["S"] * 5)
    if c["kind"] == "importance":
        nbytes += U * c["N"] * 4
    return dict(bytes=nbytes, flops=2 * c["B"] * c["L"] * c["H"] * c["W"] * c["N"] * c["d"])


def tolerance(case):
    """Four times what was seen against the same definitions in 64-bit floating point and between the
    library's two scoring modes: scores differ by up to 3e-6 (2-norm) and 5e-6 (largest), per-token
    importances by 4.3e-6 and 4.5e-5, attention outputs by 2.9e-6 and 1.2e-5; rows are copies.  Whole
    numbers differ only where two scores tie at the budget cut."""
    return {"rel": 2e-5, "max": 2e-4, "differ": 0.002}
