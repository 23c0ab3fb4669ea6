"""Rows shared by clusters of two, four and eight blocks, whose lists go to the first block as a whole: lists of hardly an entry, of odd lengths, of
many rounds of sixteen bytes, and histograms that several blocks fill in the same bins.  The rows are exchangeable and none may be handed on."""
import numpy as np
import pytest
import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


# size: blocks of a cluster (0: a few entries more, which eight do not hold).  Half of them do not hold a row's logits; twice as many would not find
# their SMs at once for the 40 and the 20 rows.
@pytest.mark.parametrize("V,K,dtype,B,W,size", [(65536, 1, wk.BF16, 1, 3, 2), (65536, 37, wk.F16, 2, 4, 2), (65536, 8192, wk.BF16, 1, 4, 2), (65528, 333, wk.F32, 1, 5, 4),
                                                (65536, 6000, wk.F32, 1, 2, 4), (131072, 4000, wk.F32, 1, 3, 8), (131064, 333, wk.F32, 1, 3, 8), (262144, 3, wk.BF16, 1, 2, 8),
                                                (262136, 4000, wk.F16, 1, 2, 8), (65536, 500, wk.BF16, 1, 40, 2), (65536, 900, wk.F32, 1, 20, 4),
                                                (131080, 4000, wk.F32, 1, 3, 0), (262152, 9000, wk.F16, 1, 2, 0)])
def test_lists_that_other_blocks_send(V, K, dtype, B, W, size):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, seed=V + K)
    p = sjd.binding.sjd_params(struct_size=sjd.binding.C.sizeof(sjd.binding.sjd_params), B=B, W=W, V=V, logits_dtype=dtype, top_k=K, stride_b=W * V,
                               stride_w=V, cfg_scale=wl.cfg_scale, inv_temperature=1.0)
    assert sjd.binding.sjd_row_path(p) == (sjd.binding.SJD_PATH_CLUSTER if size else sjd.binding.SJD_PATH_STREAM)
    assert 2 * V * (4 if dtype == wk.F32 else 2) > size // 2 * 227 * 1024
    if size and B * W > 8:
        assert B * W * 2 * size > torch.cuda.get_device_properties(0).multi_processor_count
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16)
