"""Blocks of the stream kernel that have one row, none or two: with three, two and one teams a block (by the top-K), full and ragged windows."""
import numpy as np
import pytest

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K", [(65536, 10), (65536, 2500), (65536, 18000), (50264, 300)])
@pytest.mark.parametrize("win_len", [(100, 40), (74, 74), (100, 100)])
def test_blocks_of_few_rows(V, K, win_len):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=2, W=max(win_len), V=V, top_k=K, seed=V + K)
    inp = wk.make_step_inputs(wl)
    inp.win_len = np.array(win_len, np.int32)
    p = sjd.binding.sjd_params(struct_size=sjd.binding.C.sizeof(sjd.binding.sjd_params), B=wl.B, W=wl.W, V=V, logits_dtype=wl.dtype, top_k=K,
                               stride_b=wl.W * V, stride_w=V, cfg_scale=wl.cfg_scale, inv_temperature=1.0)
    assert sjd.binding.sjd_row_path(p) == sjd.binding.SJD_PATH_STREAM
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16)
