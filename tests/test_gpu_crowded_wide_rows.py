"""Few rows with a wide top-K that lies in one block of ids: the second sift finds room for a unit's ids, so no row is redone by the any-shape path (whose
probabilities agree with the sifting kernels' to rounding only: here they are the same bits as in a call of many rows)."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K,dtype", [(65536, 8192, wk.BF16), (65536, 8192, wk.F32)])
def test_the_second_sift_takes_them(V, K, dtype):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    n = 6
    wl = wk.CONFIGS["cfg2"].scaled(B=1, W=n, V=V, top_k=K, dtype=wk.F32, seed=K, peaks=0)
    inp = wk.make_step_inputs(wl)
    for a in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond):
        a[:, :, V // 8 * 3: V // 2] += 14.0
    if dtype != wk.F32:
        inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond = (wk._store(a, dtype) for a in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond))
    inp.wl = wl.scaled(dtype=dtype)
    prev = oracle_prime(inp)
    rep, few, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert np.all(few.status & 16)  # (sifted once more)
    # the same rows over and over as sequences of one step of more rows than clusters find SMs for
    from gpu_harness import gpu_step
    kw = step_kwargs(inp)
    kw.pop("win_len"), kw.pop("pos_base")
    again = lambda a: np.concatenate([a] * 26, axis=0)
    q = type(prev.probs)(*(again(a) for a in (prev.probs.tok_prob, prev.probs.ids, prev.probs.vals, prev.probs.cnt)))
    many = gpu_step(again(inp.cond), again(inp.uncond), again(prev.tokens), q, **kw)
    assert many.vals[0].tobytes() == few.vals[0].tobytes() and many.ids[0].tobytes() == few.ids[0].tobytes()
