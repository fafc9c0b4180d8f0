"""The shot boundaries reach the kernels in the launch's parameters when they are few and through a
device copy when they are many: parity on both sides of the line (768 entries, S + 4 per prompt)."""
import pytest

import paper_2502_01941_b200 as skv
from paper_2502_01941_b200 import workloads as wl
import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = skv.Context(0)
    yield c
    c.close()


# 256 window rows so that short units stay on the single pass; chunk ends and boundaries coincide in
# the 16-token chunks, and every prompt of a batch has boundaries of its own
@pytest.mark.parametrize("B,S,lo,hi", [(1, 764, 16, 16), (1, 765, 16, 16), (4, 188, 10, 100), (4, 189, 10, 100), (3, 1, 4000, 4000)])
def test_table_in_the_parameters_and_on_the_device(ctx, B, S, lo, hi):
    N = 16 * S + 256 if lo == hi == 16 else 6000 if S == 1 else 12500
    cfg = wl.PrefillConfig("table", B=B, L=1, H=8, Hkv=2, d=64, N=N, W=64, S=S, shot_dist="uniform", shot_lo=lo, shot_hi=hi,
                           question_len=N - S * lo if lo == hi else 500, r_p=0.4, cfg_id=61)
    Q, K, V, off = wl.prefill_batch(cfg, "cuda")
    for mode in (0, 1):
        gpu = P.gpu_prefill(ctx, P.dims_of(cfg), Q, K, V, off, cfg.r_p, mode, "fused")
        assert P.check_all_units(gpu, Q, K, V, off, cfg.r_p, mode) <= 1
