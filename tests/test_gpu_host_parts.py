"""The host-buffer step in parts: every output against one sjd_step() on device copies of the same arrays."""
import numpy as np
import pytest
import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200 import binding as B_

pytestmark = pytest.mark.gpu


# (B, W, V, K, guidance): one part; parts of unequal numbers of sequences; as many parts as there may be and more
# sequences than that; fewer sequences than the bytes would make parts; long rows, in rounds; ids not 16-byte aligned.
@pytest.mark.parametrize("pinned", ["all", "none", "ids only"])
@pytest.mark.parametrize("B,W,V,K,guidance", [
    (1, 5, 512, 31, True), (5, 32, 16384, 1000, True), (19, 32, 16384, 100, True), (2, 64, 32768, 2001, False),
    (3, 16, 65536, 4099, True)])
def test_parts_equal_one_step(B, W, V, K, guidance, pinned):
    g = torch.Generator().manual_seed(B * 1000 + K)
    logits = lambda: (torch.randn(B, W, V, generator=g) * 2).to(torch.bfloat16)
    cond, uncond = logits(), logits() if guidance else None
    dev = torch.device("cuda:0")
    d_cond, d_uncond = cond.to(dev), None if uncond is None else uncond.to(dev)
    params = lambda flags, **kw: dict(cfg_scale=2.0, inv_temperature=1.25, reuse_tau=0.4, flags=flags, **kw)
    pos = torch.arange(B, dtype=torch.int32) * 7
    win = torch.tensor([W - b % 3 for b in range(B)], dtype=torch.int32)

    d_pos, d_win = pos.to(dev), win.to(dev)
    ws = torch.empty(sjd.sjd_workspace_bytes(sjd.make_params(d_cond, top_k=K)), dtype=torch.uint8, device=dev)

    # a first step drafts every row; the second one, on other logits of the same rows, verifies them
    ids = lambda *shape: torch.full(shape, -7, dtype=torch.int32, device=dev)
    acc, tok, first = ids(B), ids(B, W), sjd.DeviceProbs.empty(B, W, K, dev)
    p = sjd.make_params(d_cond, top_k=K, pos_base=d_pos, workspace=ws, **params(B_.SJD_FLAG_DRAFT_ALL))
    sjd.sjd_step(d_cond, d_uncond, None, None, p, 11, acc, tok, first)
    drafts = tok.clone()
    cond = (cond.float() + 0.7 * torch.randn(B, W, V, generator=g)).to(torch.bfloat16)
    d_cond = cond.to(dev)
    flags, status, want = ids(B, W), ids(B), sjd.DeviceProbs.empty(B, W, K, dev)
    for t in (want.ids, want.cnt):
        t.fill_(-7)
    p = sjd.make_params(d_cond, top_k=K, pos_base=d_pos, win_len=d_win, iteration0=1, out_flags=flags,
                        status=status, workspace=ws, **params(B_.SJD_FLAG_REUSE))
    sjd.sjd_step(d_cond, d_uncond, drafts, first, p, 11, acc, tok, want)
    torch.cuda.synchronize()

    pin = lambda t: t.cpu().pin_memory()
    hold = pin if pinned == "all" else lambda t: t.cpu().clone()
    h_q = sjd.HostProbs(hold(first.tok_prob), (pin if pinned != "none" else hold)(first.ids), hold(first.vals),
                        hold(first.cnt))
    h_out = sjd.HostProbs.empty(B, W, K, pin=pinned == "all")
    h_acc, h_tok, h_flags, h_status = (hold(torch.full_like(t, -9)) for t in (acc, tok, flags, status))
    ctx = sjd.HostContext(B, W, V, B_.SJD_BF16, K, device=dev)
    h_win, h_pos = hold(win), hold(pos)
    hp = ctx.params(win_len=h_win, pos_base=h_pos, iteration0=1, out_flags=h_flags, status=h_status,
                    **params(B_.SJD_FLAG_REUSE))
    for _ in range(2):  # the second call finds the first one's words in every mirror
        sjd.sjd_step_host(ctx, hold(cond), None if uncond is None else hold(uncond), hold(drafts), h_q, hp, 11, h_acc, h_tok,
                          h_out)
    ctx.close()
    live = (torch.arange(W).view(1, W) < win.view(B, 1))
    assert torch.equal(h_acc, acc.cpu()) and torch.equal(h_status, status.cpu())
    for h, d in ((h_tok, tok), (h_flags, flags), (h_out.cnt, want.cnt), (h_out.ids, want.ids)):
        assert torch.equal(h[live], d.cpu()[live])
    # fewer rows at a time may be taken by another kernel, which adds a row's exponentials up in another order: two sums
    # of K terms by 32 lanes and a tree, and a few roundings around them
    bound = 2 * (K / 32 + 8) * 2.0 ** -24
    for h, d in ((h_out.tok_prob, want.tok_prob), (h_out.vals, want.vals)):
        np.testing.assert_allclose(h[live].numpy(), d.cpu()[live].numpy(), rtol=bound, atol=0)
