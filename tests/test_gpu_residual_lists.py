"""The residual draw's look at the previous iteration's row: lists that lie anywhere against this row's, and rows without a list."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


def _inputs(V, K, W, seed):
    wl = wk.CONFIGS["cfg2"].scaled(B=2, W=W, V=V, top_k=K, seed=seed, peaks=0)
    return wl, wk.make_step_inputs(wl)


# all of the previous row's ids between two neighbours of this row's, below all of them, above all of them, every other one the same
@pytest.mark.parametrize("K", [5, 2000, 2048, 5000])
@pytest.mark.parametrize("where", ["between", "below", "above", "interleaved"])
def test_previous_ids_anywhere(K, where):
    from gpu_harness import check_parity, step_kwargs
    V, W = 65536, 4
    wl, inp = _inputs(V, K, W, K)
    # this row's largest entries: the ids [a, a + half) and [b, b + rest); the previous row's elsewhere
    half = K // 2
    a, b = {"between": (100, 40000), "below": (20000, 40000), "above": (100, 8000), "interleaved": (100, 40000)}[where]
    own = np.r_[a:a + half, b:b + K - half]
    q0 = {"between": 9000, "below": 100, "above": 50000, "interleaved": 0}[where]
    q_ids = np.arange(q0, q0 + K) if where != "interleaved" else np.unique(np.r_[own[::2], 50000 + np.arange(K)])[:K]
    for arr in (inp.cond, inp.uncond):
        f = wk._as_f32(arr, wl.dtype).copy()
        f[:, :, own] += 30.0
        arr[:] = wk._store(f, wl.dtype)
    rng = np.random.default_rng(K)
    vals = rng.random((2, W, K)).astype(np.float32)
    vals /= vals.sum(-1, keepdims=True)
    ids = np.ascontiguousarray(np.broadcast_to(q_ids.astype(np.int32), (2, W, K)))
    drafts = np.ascontiguousarray(ids[:, :, K // 2])
    q = oracle.Probs(np.ascontiguousarray(vals[:, :, K // 2]), ids, vals, np.full((2, W), K, np.int32))
    check_parity(inp.cond, inp.uncond, drafts, q, step_kwargs(inp), inp.win_len)


@pytest.mark.parametrize("K", [64, 2048, 3000])
def test_rows_without_a_list_need_none(K):
    # uniform rows in lists of a single entry: nothing of them is read
    import paper_2512_07503_b200 as sjd
    from gpu_harness import gpu_step, step_kwargs, to_device_logits
    V, W, B = 16384, 5, 2
    wl, inp = _inputs(V, K, W, K + 1)
    q = oracle.Probs.uniform(B, W, K, V)
    drafts = np.random.default_rng(K).integers(0, V, (B, W)).astype(np.int32)
    want = gpu_step(inp.cond, inp.uncond, drafts, q, **step_kwargs(inp))
    dev = "cuda:0"
    i32 = dict(dtype=torch.int32, device=dev)
    small = sjd.DeviceProbs(torch.from_numpy(q.tok_prob).to(dev), torch.zeros(1, **i32), torch.zeros(1, device=dev), torch.from_numpy(q.cnt).to(dev))
    cond, uncond = to_device_logits(inp.cond, wl.dtype), to_device_logits(inp.uncond, wl.dtype)
    out, acc, tok = sjd.DeviceProbs.empty(B, W, K, dev), torch.zeros(B, **i32), torch.zeros(B, W, **i32)
    kw = step_kwargs(inp)
    win, pos = (None if kw[k] is None else torch.from_numpy(np.ascontiguousarray(kw[k], np.int32)).to(dev) for k in ("win_len", "pos_base"))
    ws, d = torch.empty(1 << 16, dtype=torch.uint8, device=dev), torch.from_numpy(drafts).to(dev)
    p = sjd.make_params(cond, top_k=K, cfg_scale=kw["cfg_scale"], inv_temperature=kw["inv_temperature"], reuse_tau=kw["reuse_tau"], flags=kw["flags"],
                        iteration0=kw["iteration0"], win_len=win, pos_base=pos, workspace=ws)
    sjd.sjd_step(cond, uncond, d, small, p, kw["seed"], acc, tok, out)
    assert np.array_equal(acc.cpu().numpy(), want.accept_len) and np.array_equal(tok.cpu().numpy(), want.tokens)
    assert out.tok_prob.cpu().numpy().tobytes() == want.tok_prob.tobytes()
