"""More sequences than SMs (166 of 148 is the last number that the verification takes one to an SM): lists of one entry, of a round of its entries, of
several rounds, with and without probabilities in the map, without a map, uniform references among them."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,W,V,K", [(166, 1, 4096, 64), (167, 2, 4096, 1), (400, 1, 2048, 2048), (167, 1, 4096, 2049), (310, 1, 8192, 8192), (170, 1, 16384, 9001),
                                     (168, 1, 65536, 49160), (168, 1, 65544, 65537), (168, 1, 1227240, 8201), (168, 1, 1183616, 100)])
def test_many_sequences(B, W, V, K):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    n = B if V < 100000 else 2
    wl = wk.CONFIGS["cfg2"].scaled(B=n, W=W, V=V, top_k=K, seed=V + K, peaks=0, sigma=1.0)
    inp = wk.make_step_inputs(wl)
    if n < B:  # large rows: the same two for every sequence, which draws its own numbers
        of = np.arange(B) % n
        inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond, inp.win_len, inp.pos_base = (np.ascontiguousarray(a[of]) for a in (
            inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond, inp.win_len, inp.pos_base))
        inp.wl = wl.scaled(B=B)
    prev = oracle_prime(inp, n_threads=16)
    prev.probs.cnt[::5] = -1  # (these have no list)
    prev.probs.tok_prob[::5] = 1.0 / V
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len, n_threads=16)
