"""Thresholds that lie within two octaves below the largest sampled value and thresholds that do not: the sample's cuts (one, two and four vectors a
piece, one, two and four groups a vector), ranks from the first maximum to half of them, logits of both signs, of one sign, of large and of small size,
few rows and many.  A threshold that is off shows as a row that is handed on: the rows here are exchangeable and none may be."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,W", [(1, 5), (1, 160)])
@pytest.mark.parametrize("V,K", [(2048, 1), (2048, 250), (4104, 64), (16384, 16), (16384, 4000), (65536, 2000)])
# (Thresholds are bf16 numbers, lowered by half a step.  A step at the values here is at most 1 / 30 of a row's spread of 33, which passes 3 % more
# candidates; the lists have room for 20 %.  At a shift of 500 a step is an eighth of the spread: 14 % more beside the estimate's own error, and rows overrun.)
@pytest.mark.parametrize("dtype,sigma,shift", [(wk.F32, 2.0, 0.0), (wk.BF16, 2.0, -10.0), (wk.F16, 30.0, 50.0)])
def test_no_exchangeable_row_is_handed_on(B, W, V, K, dtype, sigma, shift):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    if W > 100 and V * K > 1 << 26:
        B, W = 1, 150  # (the oracle's time)
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, top_k=K, dtype=wk.F32, sigma=1.0, peaks=0, seed=V + K, cfg_scale=1.5)
    inp = wk.make_step_inputs(wl)
    for a in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond):
        a *= sigma
        a += shift
    if dtype != wk.F32:
        inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond = (wk._store(a, dtype) for a in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond))
    inp.wl = wl.scaled(dtype=dtype)
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16)
