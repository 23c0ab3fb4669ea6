"""Rows that move up in the window: their lists are copied whole, whatever their length and alignment, and nothing past them."""
import pytest
import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200 import binding as B_

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# below a vector, around one, odd (rows at every alignment), the ends of one and of two rounds of 256 threads by words and by
# vectors, and past them; offset: lists that start off a 16-byte boundary
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("K", [1, 3, 4, 6, 255, 257, 511, 513, 1000, 2044, 2048, 2052, 4102])
def test_moved_rows_keep_their_lists(K, offset):
    B, W, V, N = 2, 5, 8192, 100
    g = torch.Generator().manual_seed(K)

    def probs(fill):
        make = lambda n, dt: torch.full((n + offset + 8,), fill, dtype=dt, device=DEV)[offset:offset + n]
        f, i = torch.float32, torch.int32
        return B_.DeviceProbs(make(B * W, f).view(B, W), make(B * W * K, i).view(B, W, K), make(B * W * K, f).view(B, W, K),
                              make(B * W, i).view(B, W))
    step, nxt = probs(0), probs(-5)
    step.ids.copy_(torch.randint(0, V, (B, W, K), generator=g))
    step.vals.copy_(torch.rand(B, W, K, generator=g))
    step.tok_prob.copy_(torch.rand(B, W, generator=g))
    step.cnt.fill_(K)
    i32 = dict(dtype=torch.int32, device=DEV)
    win, pos, it = torch.full((B,), W, **i32), torch.zeros(B, **i32), torch.ones(B, **i32)
    acc = torch.tensor([1, 0], **i32)  # two rows committed, one row committed
    tok, drafts = torch.arange(B * W, **i32).view(B, W), torch.full((B, W), -3, **i32)
    committed = torch.full((B, N), -1, **i32)
    logits = torch.empty(V, dtype=torch.bfloat16, device=DEV).as_strided((B, W, V), (0, 0, 1))
    p = sjd.make_params(logits, top_k=K)
    sjd.sjd_window_advance(p, N, 3, acc, tok, step, win, pos, it, drafts, nxt, committed)
    torch.cuda.synchronize()
    for b, c in enumerate((2, 1)):
        for a, z in ((nxt.ids, step.ids), (nxt.vals, step.vals), (nxt.tok_prob, step.tok_prob), (nxt.cnt, step.cnt),
                     (drafts, tok)):
            assert torch.equal(a[b, :W - c], z[b, c:])
        assert int((nxt.ids[b, W - c:] != -5).sum()) == 0  # new random slots have no list: not written
    assert win.tolist() == [W, W] and pos.tolist() == [2, 1] and it.tolist() == [2, 2]
