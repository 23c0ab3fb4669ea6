"""The extension module's way to the library against binding.py's own: the same outputs, and the same refusals."""
import numpy as np
import pytest
import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200 import workloads as wk


class _Params(sjd.binding.sjd_params):
    """Not the ordinary type: goes through binding.py."""


def _step(inp, prev, params_type):
    from gpu_harness import DEV, probs_to_device, step_kwargs, to_device_logits
    wl, kw = inp.wl, step_kwargs(inp)
    i32 = dict(dtype=torch.int32, device=DEV)
    cond, uncond = to_device_logits(inp.cond, wl.dtype), to_device_logits(inp.uncond, wl.dtype)
    out, acc, tok = sjd.DeviceProbs.empty(wl.B, wl.W, wl.kcap, DEV), torch.zeros(wl.B, **i32), torch.zeros(wl.B, wl.W, **i32)
    p = sjd.make_params(cond, top_k=wl.top_k, cfg_scale=kw["cfg_scale"], flags=kw["flags"], iteration0=1)
    ws = torch.empty(sjd.sjd_workspace_bytes(p), dtype=torch.uint8, device=DEV)
    p.workspace, p.workspace_bytes = ws.data_ptr(), ws.numel()
    q = params_type.from_buffer_copy(p)
    q._keepalive = (ws, p)  # (the copy has the address only)
    args = [cond, uncond, torch.from_numpy(prev.tokens).to(DEV), probs_to_device(prev.probs), q, kw["seed"], acc, tok, out]
    return args, lambda: [t.cpu().numpy().tobytes() for t in (acc, tok, out.tok_prob, out.ids, out.vals, out.cnt)]


@pytest.mark.gpu
def test_both_ways_give_the_same_and_refuse_the_same():
    from gpu_harness import oracle_prime
    wl = wk.CONFIGS["cfg1"]
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    got = []
    for kind in (sjd.binding.sjd_params, _Params):
        args, read = _step(inp, prev, kind)
        before = sjd.sjd_launch_count()
        sjd.sjd_step(*args)
        assert sjd.sjd_launch_count() == before + 2
        got.append(read())
        wrong = [(1, args[1].transpose(0, 1)), (2, args[2].long()), (2, args[2].cpu()), (6, args[6].float()), (7, args[7].expand(2, -1, -1)[:, :, ::2]),
                 (3, sjd.DeviceProbs(args[3].tok_prob, args[3].ids.float(), args[3].vals, args[3].cnt)), (0, args[0].cpu())]
        for at, value in wrong:
            with pytest.raises(sjd.binding.SjdError):
                sjd.sjd_step(*args[:at], value, *args[at + 1:])
        with pytest.raises(sjd.binding.SjdError):  # refused by the library itself
            sjd.sjd_step(*args[:6], None, *args[7:])
        sjd.sjd_step(*args[:5], np.int64(args[5]), *args[6:])  # (a number of another type)
        assert read() == got[-1]
        assert sjd.sjd_launch_count() == before + 4
    assert got[0] == got[1]


@pytest.mark.gpu
@pytest.mark.parametrize("counted", [True, False])
def test_both_ways_advance_the_window_alike(counted):
    from gpu_harness import DEV, oracle_prime
    inp = wk.make_step_inputs(wk.CONFIGS["cfg1"].scaled(B=3))
    wl, prev, n_total = inp.wl, oracle_prime(inp), 40
    got = []
    for kind in (sjd.binding.sjd_params, _Params):
        args, _ = _step(inp, prev, kind)
        sjd.sjd_step(*args)
        acc, tok, out, p = args[6], args[7], args[8], args[4]
        i32 = dict(dtype=torch.int32, device=DEV)
        win, pos, it = torch.tensor([16, 9, 4], **i32), torch.tensor([0, 31, 36], **i32), torch.tensor([1, 2, 5], **i32)
        drafts, nxt = torch.full((wl.B, wl.W), -7, **i32), sjd.DeviceProbs.empty(wl.B, wl.W, wl.kcap, DEV)
        committed, count = torch.full((wl.B, n_total), -7, **i32), torch.full((wl.B,), -7, **i32)
        before = sjd.sjd_launch_count()
        sjd.sjd_window_advance(p, n_total, 77, acc, tok, out, win, pos, it, drafts, nxt, committed, count if counted else None)
        assert sjd.sjd_launch_count() == before + 2
        got.append([t.cpu().numpy().tobytes() for t in (win, pos, it, drafts, nxt.tok_prob, nxt.ids, nxt.vals, nxt.cnt, committed, count)])
        assert (count.cpu().numpy() > 0).all() == counted and pos.cpu().tolist() != [0, 31, 36]
    assert got[0] == got[1]


def test_refusals_without_a_gpu():
    p = sjd.binding.sjd_params()
    with pytest.raises(sjd.binding.SjdError, match="CUDA device"):
        sjd.sjd_step(torch.zeros(1, 1, 8), None, None, None, p, 0, None, None, None)
    with pytest.raises(sjd.binding.SjdError):
        sjd.sjd_window_advance(p, 4, 0, torch.zeros(1), torch.zeros(1, 1, dtype=torch.int32), *[sjd.DeviceProbs.empty(1, 1, 1, "cpu")], *[None] * 4,
                               sjd.DeviceProbs.empty(1, 1, 1, "cpu"), None)
