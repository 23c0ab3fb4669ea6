"""Rows whose K-th largest entry shares its bin of the histogram with many others (a few entries far above the rest stretch the bins): up to 32 members,
some more than that, hundreds with few different values, and more than are ranked there; the threshold at a zero of either sign."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu

V = 16384


@pytest.mark.parametrize("B,W", [(1, 4), (1, 160)])
# the distance to the largest entries; entries of the bin come to about a twelfth of the first, of values a sixteenth apart
@pytest.mark.parametrize("K,top", [(40, 8.0), (100, 30.0), (300, 30.0), (2000, 30.0), (300, 1000.0), (1000, 1000.0), (2000, 1000.0)])
@pytest.mark.parametrize("dtype", [wk.F32, wk.BF16])
def test_members_of_the_threshold_bin(B, W, K, top, dtype):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, top_k=K, dtype=dtype, cfg_scale=1.0, seed=K)
    inp = wk.make_step_inputs(wl)
    rng = np.random.Generator(np.random.Philox(K))

    def logits():
        x = rng.standard_normal((B, W, V), dtype=np.float32)
        x -= np.sort(x, axis=2)[:, :, V - K, None]  # the K-th largest is zero
        x = np.round(x * 16) / np.float32(16)
        x *= np.where(rng.random(x.shape) < 0.5, np.float32(-1), np.float32(1)) ** (x == 0)  # zeros of both signs
        x[:, :, [5, 7777, V - 1]] = top
        return wk._store(x, dtype)

    inp.cond, inp.prev_cond, inp.uncond, inp.prev_uncond = logits(), logits(), None, None
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, None, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert np.all(got.cnt == K)
