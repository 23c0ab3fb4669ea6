"""Rows shared by clusters of two, four and eight blocks, whose lists go to the first block as a whole: lists of hardly an entry, of odd lengths, of
many rounds of sixteen bytes, and histograms that several blocks fill in the same bins.  The rows are exchangeable and none may be handed on."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K,dtype,B,W", [(65536, 1, wk.BF16, 1, 3), (65536, 37, wk.F16, 2, 4), (65536, 8192, wk.BF16, 1, 4), (65528, 333, wk.F32, 1, 5),
                                           (65536, 6000, wk.F32, 1, 2), (131080, 4000, wk.F32, 1, 3), (262144, 3, wk.BF16, 1, 2), (262152, 9000, wk.F16, 1, 2)])
def test_lists_that_other_blocks_send(V, K, dtype, B, W):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, seed=V + K)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16)
