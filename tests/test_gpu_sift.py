"""GPU parity of the row kernels that sift a row by a sampled threshold, at the sizes where their cutting of a row can
go wrong: vocabularies around a segment, a unit and half a unit, few rows (clusters of 8, 4, 2 and 1 CTAs) and many
(teams sharing a ring), top-K from 1 to 8,192, every logits type."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


def _check(name, **over):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(name=name, **over)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16), "an ordinary row was redone by the any-shape path"
    return inp, prev, wl


@pytest.mark.parametrize("dtype", [wk.BF16, wk.F16, wk.F32])
@pytest.mark.parametrize("V", [2048, 2056, 4088, 8200, 16376, 16392])
@pytest.mark.parametrize("B,W", [(1, 1), (3, 7), (2, 30), (1, 140), (9, 33)])
def test_cutting_of_a_row(V, B, W, dtype):
    _check(f"cut{V}", B=B, W=W, V=V, dtype=dtype, top_k=1 + V // 40, seed=V + W, ragged_total=0 if B > 1 else 24)


@pytest.mark.parametrize("V,K,B,W", [(50264, 2000, 1, 8), (65536, 4096, 1, 5), (65536, 8192, 2, 76), (32776, 1, 2, 3),
                                     (131072, 3000, 1, 2), (20000, 5000, 1, 3),
                                     (65536, 9001, 1, 6), (65536, 2049, 3, 2)])
def test_wide_rows_and_wide_top_k(V, K, B, W):
    _check(f"wide{V}", B=B, W=W, V=V, top_k=K, seed=K + W)


@pytest.mark.parametrize("B,W", [(1, 3), (2, 80)])
def test_rows_whose_lists_run_over_are_redone(B, W):
    # everything but the sample's pieces is large: too many entries reach the sampled threshold
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    V = 10008
    wl = wk.CONFIGS["cfg1"].scaled(B=B, W=W, V=V, top_k=100)
    inp = wk.make_step_inputs(wl)
    stride = ((V + 255) // 256 + 7) // 8 * 8
    sampled = (np.arange(V) % stride) < 16
    for arr in (inp.cond, inp.uncond):
        arr[:, 0, sampled] -= 50.0
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert np.all(got.status & 16)
