"""What the performance of this library is measured on.

Every case is one of three things a program does with the library:

* ``step``  one verify-and-redraft step on logits that lie on the device (``sjd_step``), or the draft of a
            first window from predicted distributions (``SJD_FLAG_DRAFT_ALL``);
* ``loop``  a stretch of the decode loop of an image (``DecodeLoop.run``), the model replaced by logits that
            are ready on the device;
* ``host``  one step on pinned host buffers (``sjd_step_host``), copies in and out included.

The sizes are those of the configurations and sweep shapes in ``paper_2512_07503_b200/workloads.py``, and
generic ones beside them where real use has other vocabularies, windows and settings.
"""
import math

import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200.decode import DecodeLoop

DEVICE = "cuda:0"
DTYPES = {"f32": (torch.float32, 0, 4), "bf16": (torch.bfloat16, 1, 2), "f16": (torch.float16, 2, 2)}

_BASE = dict(kind="step", B=1, W=32, V=65536, dtype="bf16", top_k=2000, guidance=True, scale=3.0, temperature=1.0,
             reuse=True, draft_all=False, sigma=3.0, peaks=20, boost=8.0, grid=0, iterations=0, init_mode=0)


def _case(**kw):
    return dict(_BASE, **kw)


def listed():
    return [
        # the smallest call: one short window, a small vocabulary, fp32 logits
        _case(name="step_small", B=1, W=16, V=4096, dtype="f32", top_k=64, sigma=2.0, peaks=0),
        # one image at a time: a single window over the full vocabulary
        _case(name="step_one_image", B=1, W=32),
        # a serving batch whose sequences stand at different places of a 24 x 24 grid: ragged windows, fp32
        # logits, another guidance scale and a temperature
        _case(name="step_ragged_f32", B=64, W=16, V=16384, dtype="f32", top_k=1000, scale=4.0, temperature=0.9,
              sigma=2.5, peaks=10, boost=6.0, grid=576),
        # the headline: sixteen images, window 64, full vocabulary, bf16
        _case(name="step_batch", B=16, W=64),
        # long odd windows, fp16 logits, a small top-K
        _case(name="step_window250_f16", B=4, W=250, dtype="f16", top_k=100),
        # the small image vocabulary with the same top-K: much selection per byte
        _case(name="step_v16k", B=16, W=64, V=16384),
        # a wide top-K
        _case(name="step_k8192", B=16, W=64, top_k=8192),
        # first windows drafted from predicted distributions, a model without guidance, with a temperature
        _case(name="draft_no_guidance", B=32, W=32, V=32768, guidance=False, temperature=0.8, draft_all=True),
        # a vocabulary that is no power of two (text and image tokens in one head), odd batch and window,
        # plain refinement without reuse
        _case(name="step_odd_vocab", B=7, W=33, V=50264, dtype="bf16", top_k=500, scale=1.5, reuse=False),
        # decode loop of one image: step, commit, shift and refill, random initialisation of new slots
        _case(name="loop_one_image", kind="loop", B=1, W=32, grid=2304, iterations=32),
        # decode loop of a batch on a 24 x 24 grid, new slots drawn from the prediction above them
        _case(name="loop_batch_f16", kind="loop", B=16, W=16, V=16384, dtype="f16", top_k=1000, grid=576, iterations=16,
              init_mode=4),
        # logits that come from another process or machine in host memory
        _case(name="host_step", kind="host", B=4, W=32, V=16384, top_k=1000),
    ]


def draw(rng):
    """One more case of the ranges above: vocabularies of 4,096 to 65,536 entries (round ones and multiples of 8),
    windows of 1 to 250 rows, batches up to 64, at most as many logits in a call as the headline's."""
    kind = rng.choice(["step"] * 7 + ["loop"] * 2 + ["host"])
    logv = rng.uniform(math.log(4096), math.log(65536))
    V = rng.choice([4096, 8192, 16384, 32768, 65536, 65536, 16384]) if rng.random() < 0.6 else 8 * round(math.exp(logv) / 8)
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    K = min(V // 8, round(math.exp(rng.uniform(0.0, math.log(2000))))) if rng.random() < 0.5 else min(V // 8, rng.choice([100, 500, 1000, 2000]))
    if kind == "step":
        rows = min(round(math.exp(rng.uniform(0.0, math.log(1024)))), (1 << 27) // V // DTYPES[dtype][2])
        W = rng.randint(1, max(1, min(250, rows)))
        B = max(1, min(64, rows // W))
        if rng.random() < 0.15 and V >= 32768:
            K = rng.choice([4096, 5000, 8192]) if V == 65536 else 4096
        iterations = 0
    elif kind == "loop":
        B, W = rng.choice([(1, 16), (1, 32), (1, 64), (2, 24), (4, 16), (8, 16), (3, 17)])
        iterations = rng.randint(8, 24)
    else:
        B, W = rng.choice([(1, 16), (1, 32), (2, 24), (4, 16), (3, 11)])
        V, iterations = min(V, 32768), 0
        K = min(K, V // 8)
    guidance = rng.random() < 0.8
    return _case(kind=kind, B=B, W=W, V=V, dtype=dtype, top_k=max(1, K), guidance=guidance,
                 scale=rng.choice([1.5, 3.0, 4.0, 7.5]) if guidance else 1.0, temperature=rng.choice([1.0, 1.0, 0.8, 1.2]),
                 reuse=rng.random() < 0.8, draft_all=kind == "step" and rng.random() < 0.15, sigma=rng.choice([2.0, 3.0, 3.0]),
                 peaks=rng.choice([0, 10, 20]), boost=rng.choice([6.0, 8.0]),
                 grid={"loop": 2304, "step": rng.choice([0, 0, 576]), "host": 0}[kind], iterations=iterations,
                 init_mode=rng.choice([0, 0, 1, 2, 3, 4]) if kind == "loop" else 0)


# ----------------------------------------------------------------------------------------------------------
def _logits(case, g, rows_alike=False):
    """cond and uncond logits in the storage type: Gaussian rows with a few strong tokens, uncond = cond + N(0, 1).
    rows_alike: the rows of the batch share a common part, so that drafts survive from one iteration to the next."""
    B, W, V = case["B"], case["W"], case["V"]
    dt = DTYPES[case["dtype"]][0]
    if rows_alike:
        cond = (torch.randn(B, 1, V, generator=g, device=DEVICE) * case["sigma"]).repeat(1, W, 1)
        cond += 0.3 * torch.randn(B, W, V, generator=g, device=DEVICE)
    else:
        cond = torch.randn(B, W, V, generator=g, device=DEVICE) * case["sigma"]
    if case["peaks"]:
        where = torch.randint(0, V, (B, 1 if rows_alike else W, case["peaks"]), generator=g, device=DEVICE)
        where = where.expand(B, W, case["peaks"]).contiguous()
        cond.scatter_add_(2, where, torch.full(where.shape, case["boost"], device=DEVICE))
    uncond = (cond + torch.randn(B, W, V, generator=g, device=DEVICE)).to(dt) if case["guidance"] else None
    return cond.to(dt), uncond


def _noisy(t, g):
    """The previous iteration's logits: the current ones + N(0, 0.5^2)."""
    return None if t is None else (t.float() + 0.5 * torch.randn(t.shape, generator=g, device=DEVICE)).to(t.dtype)


def _windows(case, g):
    """Valid rows and first position of every sequence: staggered over the grid where there is one."""
    B, W = case["B"], case["W"]
    if case["grid"]:
        start = torch.randint(0, case["grid"], (B,), generator=g, device=DEVICE, dtype=torch.int32)
        return torch.clamp(case["grid"] - start, max=W).to(torch.int32), start
    return torch.full((B,), W, dtype=torch.int32, device=DEVICE), torch.zeros(B, dtype=torch.int32, device=DEVICE)


def _prepare_step(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    B, W, kcap = case["B"], case["W"], min(case["top_k"], case["V"])
    s = {"case": case, "seed": seed}
    s["cond"], s["uncond"] = _logits(case, g)
    win_len, pos_base = _windows(case, g)
    s["q"], s["out"] = sjd.DeviceProbs.empty(B, W, kcap, DEVICE), sjd.DeviceProbs.empty(B, W, kcap, DEVICE)
    i32 = dict(dtype=torch.int32, device=DEVICE)
    s["drafts"], s["tokens"] = torch.zeros(B, W, **i32), torch.zeros(B, W, **i32)
    s["accept_len"], s["flags"], s["status"] = torch.zeros(B, **i32), torch.zeros(B, W, **i32), torch.zeros(B, **i32)
    common = dict(top_k=case["top_k"], cfg_scale=case["scale"], inv_temperature=1.0 / case["temperature"], win_len=win_len,
                  pos_base=pos_base, status=s["status"])
    p = sjd.make_params(s["cond"], flags=sjd.binding.SJD_FLAG_DRAFT_ALL, iteration0=0, **common)
    ws = torch.empty(sjd.sjd_workspace_bytes(p), dtype=torch.uint8, device=DEVICE)
    if not case["draft_all"]:
        # the previous iteration: every row drawn from logits a little off this iteration's
        p = sjd.make_params(s["cond"], flags=sjd.binding.SJD_FLAG_DRAFT_ALL, iteration0=0, workspace=ws, **common)
        sjd.sjd_step(_noisy(s["cond"], g), _noisy(s["uncond"], g), None, None, p, seed, s["accept_len"], s["drafts"], s["q"])
    flags = (sjd.binding.SJD_FLAG_REUSE if case["reuse"] else 0) | (sjd.binding.SJD_FLAG_DRAFT_ALL if case["draft_all"] else 0)
    s["params"] = sjd.make_params(s["cond"], flags=flags, iteration0=1, out_flags=s["flags"], workspace=ws, **common)
    return s


def _run_step(s):
    sjd.sjd_step(s["cond"], s["uncond"], s["drafts"], s["q"], s["params"], s["seed"], s["accept_len"], s["tokens"], s["out"])
    o = s["out"]
    return [s["accept_len"], s["tokens"], s["flags"], s["status"], o.tok_prob, o.ids, o.vals, o.cnt]


def _prepare_loop(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    # two iterations' logits that differ a little, used in turn: what a model gives while its prefix settles
    first = _logits(case, g, rows_alike=True)
    return {"case": case, "seed": seed, "logits": [first, (_noisy(first[0], g), _noisy(first[1], g))]}


def _run_loop(s):
    case, logits = s["case"], s["logits"]
    loop = DecodeLoop(batch=case["B"], window=case["W"], vocab=case["V"], n_total=case["grid"],
                      logits_dtype=DTYPES[case["dtype"]][0], top_k=case["top_k"], cfg_scale=case["scale"],
                      inv_temperature=1.0 / case["temperature"], reuse=case["reuse"], seed=s["seed"],
                      init_mode=case["init_mode"], grid_width=math.isqrt(case["grid"]), guidance=case["guidance"], device=DEVICE)
    committed, steps, counts = loop.run(lambda d: logits[d.steps % 2], max_steps=case["iterations"])
    q = loop.q[loop.cur]
    return [committed, counts, loop.window_tokens, loop.win_len, loop.pos_base, loop.iteration, loop.status, loop.toks,
            loop.out.ids, loop.out.vals, q.tok_prob, q.ids, q.vals, q.cnt]


def _prepare_host(case, seed):
    s = _prepare_step(dict(case, grid=0), seed)
    host = lambda t: None if t is None else t.cpu().pin_memory()
    h = {"case": case, "seed": seed}
    h["ctx"] = sjd.HostContext(case["B"], case["W"], case["V"], DTYPES[case["dtype"]][1], case["top_k"], device=DEVICE)
    h["cond"], h["uncond"], h["drafts"] = host(s["cond"]), host(s["uncond"]), host(s["drafts"])
    q = s["q"]
    h["q"] = sjd.HostProbs(host(q.tok_prob), host(q.ids), host(q.vals), host(q.cnt))
    h["out"] = sjd.HostProbs.empty(case["B"], case["W"], min(case["top_k"], case["V"]))
    h["accept_len"], h["tokens"] = host(s["accept_len"]), host(s["tokens"])
    h["status"] = host(s["status"])
    win_len, pos_base = _windows(dict(case, grid=0), None)
    h["win_len"], h["pos_base"] = host(win_len), host(pos_base)
    h["params"] = h["ctx"].params(cfg_scale=case["scale"], inv_temperature=1.0 / case["temperature"],
                                  flags=sjd.binding.SJD_FLAG_REUSE if case["reuse"] else 0, iteration0=1,
                                  win_len=h["win_len"], pos_base=h["pos_base"], status=h["status"])
    return h


def _run_host(h):
    sjd.sjd_step_host(h["ctx"], h["cond"], h["uncond"], h["drafts"], h["q"], h["params"], h["seed"], h["accept_len"],
                      h["tokens"], h["out"])
    o = h["out"]
    return [h["accept_len"], h["tokens"], h["status"], o.tok_prob, o.ids, o.vals, o.cnt]


def prepare(case, seed):
    return {"step": _prepare_step, "loop": _prepare_loop, "host": _prepare_host}[case["kind"]](case, seed)


def run(state):
    return {"step": _run_step, "loop": _run_loop, "host": _run_host}[state["case"]["kind"]](state)


def work(case):
    """Each logit read once, the sparse distributions and per-position results written once, one row of the
    previous iteration's distributions read per sequence; in a loop also the window's distributions moved up.
    Per logit: difference, multiply-add and a comparison; per survivor: the exponential, the sum and the scaling."""
    rows, V, kcap = case["B"] * case["W"], case["V"], min(case["top_k"], case["V"])
    arrays = 2 if case["guidance"] else 1
    nbytes = rows * (arrays * V * DTYPES[case["dtype"]][2] + 8 * kcap + 16)
    if not case["draft_all"]:
        nbytes += case["B"] * 8 * kcap
    flops = rows * (4 * V + 10 * kcap)
    if case["kind"] == "host":
        nbytes += rows * 8 * kcap  # the previous iteration's distributions come in whole
    if case["kind"] == "loop":
        nbytes = case["iterations"] * (nbytes + rows * 16 * kcap)
        flops *= case["iterations"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Probabilities against a softmax of 64-bit logits over the same support, on the listed shapes: 5e-8 to 4e-7 in
    the 2-norm, 2e-7 to 3e-6 at the largest; stated here is about four times the worst.  Tokens, ids and counts are
    the same except where a decision lies within rounding of its boundary (a draw next to a step of the
    distribution, a ratio next to its uniform): the share that the tests allow."""
    return {"rel": 2e-6, "max": 1.2e-5, "differ": 2e-3}
