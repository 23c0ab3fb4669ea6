"""The residual draw's map of the previous iteration's ids at the edges of its range: vocabularies of less than a word of ids, the largest that shared
memory holds a map of (with and without probabilities) and the first beyond it, lists of one entry, of a round of the kernel's entries, of several rounds, and longer than the map's
positions."""
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K", [(8, 8), (40, 33), (4096, 1), (65536, 2047), (65536, 2048), (65536, 2049), (131072, 8192), (131072, 8201), (16384, 16384),
                                 (65536, 49155), (131072, 65536), (131072, 65537), (1183608, 2048), (1183616, 2048), (1052280, 8201), (1052288, 8201), (1227240, 8201), (1240000, 8201)])
def test_map_of_the_previous_ids_at_its_edges(V, K):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    n = 3 if V < 200000 else 1
    wl = wk.CONFIGS["cfg2"].scaled(B=n, W=n, V=V, top_k=K, seed=V + K, peaks=0, sigma=1.0)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
