"""Windows that have shrunk or closed in a batch of more rows than the GPU has SMs: blocks of the row kernel whose rows all lie
beyond their windows finish at once, and their rows' results are the empty ones."""
import numpy as np
import pytest
import torch

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# A step of these sizes takes tens of microseconds; a bounded on-chip wait that runs out takes a second.
LIMIT_MS = 50.0


def _windows(kind, B, W):
    win = np.full(B, W, np.int32)
    if kind == "two at their end":
        win[6], win[8] = W - 1, 0
    elif kind == "one left":
        win[:] = 0
        win[B // 2] = 3
    elif kind == "all closed":
        win[:] = 0
    elif kind == "tail":
        win[:] = np.maximum(1, W // 10)
    return win


@pytest.mark.parametrize("dtype,V,K,B,W", [(wk.BF16, 16384, 200, 16, 16), (wk.F32, 4096, 64, 1, 200), (wk.F16, 8192, 3000, 12, 40)])
@pytest.mark.parametrize("kind", ["two at their end", "one left", "all closed", "tail"])
def test_short_windows_are_right_and_quick(kind, dtype, V, K, B, W):
    from gpu_harness import check_parity, oracle_prime, step_kwargs, to_device_logits
    import paper_2512_07503_b200 as sjd
    if kind == "two at their end" and B < 9:
        pytest.skip("needs nine sequences")
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, top_k=K, dtype=dtype, seed=V + W)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    win = _windows(kind, B, W)
    kw = step_kwargs(inp, win_len=win)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, kw, win)
    dead = np.arange(W)[None, :] >= win[:, None]
    assert np.all(got.cnt[dead] == 0) and np.all(got.tokens[dead] == -1) and np.all(got.flags[dead] == 0)

    cond, uncond = to_device_logits(inp.cond, dtype), to_device_logits(inp.uncond, dtype)
    i32 = dict(dtype=torch.int32, device=DEV)
    win_d, acc, tok = torch.from_numpy(win).to(DEV), torch.zeros(B, **i32), torch.zeros(B, W, **i32)
    out = sjd.DeviceProbs.empty(B, W, K, DEV)
    ws = torch.empty(1 << 20, dtype=torch.uint8, device=DEV)
    p = sjd.make_params(cond, top_k=K, win_len=win_d, flags=sjd.binding.SJD_FLAG_DRAFT_ALL, workspace=ws)
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(2):  # the second one counts
        begin.record()
        sjd.sjd_step(cond, uncond, None, None, p, 3, acc, tok, out)
        end.record()
        torch.cuda.synchronize()
    assert begin.elapsed_time(end) < LIMIT_MS


def test_batched_decode_to_the_last_token_has_no_slow_iteration():
    # sequences of a batch finish one after the other; the last ones leave most blocks without a live row
    from paper_2512_07503_b200.decode import DecodeLoop
    B, W, V, N = 16, 16, 4096, 576
    g = torch.Generator(device=DEV).manual_seed(1)
    base = torch.randn(B, 1, V, generator=g, device=DEV) * 3
    logits = [(base + 0.5 * torch.randn(B, W, V, generator=g, device=DEV)).to(torch.bfloat16) for _ in range(3)]
    loop = DecodeLoop(batch=B, window=W, vocab=V, n_total=N, logits_dtype=torch.bfloat16, top_k=100, seed=4, device=DEV)
    events = []

    def source(d):
        if len(events) < 3 * N:
            events.append(torch.cuda.Event(enable_timing=True))
            events[-1].record()
        return logits[d.steps % 3], logits[(d.steps + 1) % 3]

    committed, steps, counts = loop.run(source, max_steps=3 * N)
    assert int(counts.sum()) == B * N and int(committed.min()) >= 0
    finished = (counts.cumsum(0) >= N).float().argmax(0)
    assert finished.min() < finished.max()  # (they do end apart)
    times = sorted(a.elapsed_time(b) for a, b in zip(events[1:], events[2:]))
    print("iterations", steps, "median", times[len(times) // 2], "ms, longest", times[-1], "ms")
    assert times[-1] < LIMIT_MS
