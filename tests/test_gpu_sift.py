"""GPU parity of the row kernels that sift a row by a sampled threshold, at the sizes where their cutting of a row can
go wrong: vocabularies around a segment, a unit and half a unit, few rows (clusters of 8, 4, 2 and 1 CTAs) and many
(teams sharing a ring), top-K from 1 to 8,192, every logits type."""
import numpy as np
import pytest

from paper_2512_07503_b200 import workloads as wk

pytestmark = pytest.mark.gpu


def _check(name, **over):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(name=name, **over)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16), "an ordinary row was redone by the any-shape path"
    return inp, prev, wl


@pytest.mark.parametrize("dtype", [wk.BF16, wk.F16, wk.F32])
@pytest.mark.parametrize("V", [2048, 2056, 4088, 8200, 16376, 16392])
@pytest.mark.parametrize("B,W", [(1, 1), (3, 7), (2, 30), (1, 140), (9, 33)])
def test_cutting_of_a_row(V, B, W, dtype):
    _check(f"cut{V}", B=B, W=W, V=V, dtype=dtype, top_k=1 + V // 40, seed=V + W, ragged_total=0 if B > 1 else 24)


def test_more_rows_than_one_launch_takes():
    _check("launches", B=20, W=500, V=2048, top_k=9, seed=11)


@pytest.mark.parametrize("V,K,B,W", [(50264, 2000, 1, 8), (65536, 4096, 1, 5), (65536, 8192, 2, 76), (32776, 1, 2, 3),
                                     (131072, 3000, 1, 2), (20000, 5000, 1, 3),
                                     (65536, 9001, 1, 6), (65536, 2049, 3, 2)])
def test_wide_rows_and_wide_top_k(V, K, B, W):
    _check(f"wide{V}", B=B, W=W, V=V, top_k=K, seed=K + W)


@pytest.mark.parametrize("B,W", [(1, 3), (2, 80)])
def test_rows_whose_lists_run_over_are_redone(B, W):
    # everything but the sample's pieces is large: too many entries reach the sampled threshold
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    V = 10008
    wl = wk.CONFIGS["cfg1"].scaled(B=B, W=W, V=V, top_k=100)
    inp = wk.make_step_inputs(wl)
    stride = ((V + 255) // 256 + 7) // 8 * 8
    sampled = (np.arange(V) % stride) < 16
    for arr in (inp.cond, inp.uncond):
        arr[:, 0, sampled] -= 50.0
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert np.all(got.status & 16)


def test_a_copy_that_never_lands_becomes_a_status_word_among_many_rows(tmp_path):
    # as tests/test_gpu_timeout.py, for the kernel whose teams share a ring: CTAs with a second row lose one of its copies
    import os
    import subprocess
    import sys
    from paper_2512_07503_b200 import build
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    lib = build.build_variant(str(tmp_path / "libsjd_timeout_rows.so"), ["SJD_TEST_SPIN_CYCLES=2000000", "SJD_TEST_DROP_COPY=3"])
    script = """
import sys
sys.path.insert(0, %r); sys.path.insert(0, %r)
import numpy as np, torch, oracle
from paper_2512_07503_b200 import workloads as wk
from gpu_harness import gpu_step, step_kwargs
wl = wk.CONFIGS["cfg2"].scaled(B=4, W=100, V=16384, top_k=200)
inp = wk.make_step_inputs(wl)
kw = step_kwargs(inp, flags=oracle.FLAG_DRAFT_ALL, iteration0=0)
for _ in range(2):
    got = gpu_step(inp.cond, inp.uncond, None, None, **kw)
    lost = got.cnt == 0
    assert np.any(lost) and np.any(~lost), lost.sum()
    assert np.array_equal(np.any(lost, axis=1), (got.status & 8) != 0)
assert torch.arange(10, device="cuda:0").sum().item() == 45
print("ROWS_TIMEOUT_OK")
""" % (root, os.path.join(root, "tests"))
    out = subprocess.run([sys.executable, "-c", script], env=dict(os.environ, SJD_LIBRARY=lib), capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and "ROWS_TIMEOUT_OK" in out.stdout, out.stdout[-2000:] + out.stderr[-4000:]


@pytest.mark.parametrize("scale,temperature", [(3.0, 1.0), (7.5, 0.8), (1.0, 1.0), (3.1, 1.3), (0.0, 1.0)])
@pytest.mark.parametrize("dtype", [wk.BF16, wk.F16])
@pytest.mark.parametrize("B,W", [(1, 4), (2, 90)])
def test_screening_keeps_what_cancels(B, W, dtype, scale, temperature):
    # the merged logit is a small difference of large ones, and some unconditional logits exceed everything the sample
    # shows: what the packed 16-bit screening must not lose
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=8192, dtype=dtype, top_k=150, cfg_scale=scale, temperature=temperature, seed=W)
    inp = wk.make_step_inputs(wl)
    rng = np.random.default_rng(W + dtype)
    shape = inp.cond.shape
    y = rng.standard_normal(shape).astype(np.float32) * 3
    u = rng.standard_normal(shape).astype(np.float32) * 40
    u[rng.random(shape) < 0.003] *= 30
    c = u + (y - u) / scale if scale else u + y
    for arr, x in ((inp.cond, c), (inp.uncond, u), (inp.prev_cond, c + 0.5), (inp.prev_uncond, u)):
        arr[:] = wk._store(x.astype(np.float32), dtype)
    prev = oracle_prime(inp)
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)


@pytest.mark.parametrize("unit", [1e-36, 3e-38, 1e-40])
@pytest.mark.parametrize("B,W", [(1, 3), (2, 90)])
def test_rows_whose_candidates_differ_by_next_to_nothing(B, W, unit):
    # a few hundred entries between 0 and `unit` (normal and subnormal numbers), everything else at -1: the candidates' bins
    # are as narrow as floats allow, and the threshold lies among them
    from gpu_harness import check_parity, step_kwargs
    wl = wk.CONFIGS["cfg1"].scaled(B=B, W=W, V=4096, top_k=64, seed=W)
    inp = wk.make_step_inputs(wl)
    rng = np.random.default_rng(W)
    for arr in (inp.cond, inp.prev_cond):
        arr[:] = -1.0
        pick = rng.random(arr.shape) < 0.15
        arr[pick] = (rng.random(int(pick.sum())) * unit).astype(np.float32)
    prev = _prime_without_guidance(inp)
    check_parity(inp.cond, None, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)


def _prime_without_guidance(inp):
    import oracle
    from gpu_harness import step_kwargs
    kw = step_kwargs(inp, flags=oracle.FLAG_DRAFT_ALL, iteration0=inp.iteration - 1)
    return oracle.sjd_step(inp.prev_cond, None, None, None, V=inp.wl.V, n_threads=8, diag=True, **kw)


@pytest.mark.parametrize("dtype,u_size,c_size", [(wk.BF16, 1e7, 3.0), (wk.BF16, 1e5, 0.03), (wk.F16, 6e4, 0.01), (wk.BF16, 3e3, 3.0)])
@pytest.mark.parametrize("B,W", [(1, 4), (2, 90)])
def test_screening_keeps_what_32_bit_rounding_lifts(B, W, dtype, u_size, c_size):
    # guidance scale 1: the merged logit is c - u + u, off from c by 2^-24 of a |u| that dwarfs the threshold
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=16384, dtype=dtype, top_k=150, cfg_scale=1.0, seed=W)
    inp = wk.make_step_inputs(wl)
    rng = np.random.default_rng(W + dtype)
    shape = inp.cond.shape
    c = rng.standard_normal(shape).astype(np.float32) * c_size
    u = np.clip(rng.standard_normal(shape).astype(np.float32), -1, 1) * u_size
    for arr, x in ((inp.cond, c), (inp.uncond, u), (inp.prev_cond, c + c_size / 8), (inp.prev_uncond, u)):
        arr[:] = wk._store(x.astype(np.float32), dtype)
    prev = oracle_prime(inp)
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)


@pytest.mark.parametrize("mask", ["a tenth in one piece", "every other token"])
@pytest.mark.parametrize("V,K,dtype,B,W,temperature", [(65536, 2000, wk.BF16, 2, 76, 1.0), (50264, 500, wk.BF16, 1, 6, 0.8),
                                                       (50264, 500, wk.F16, 3, 53, 1.0), (16384, 300, wk.F32, 2, 80, 1.0)])
def test_masked_tokens_are_no_candidates(V, K, dtype, B, W, temperature, mask):
    # tokens forbidden with -inf in both arrays: their merge is a NaN, and no row is redone for them
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, temperature=temperature, seed=W)
    inp = wk.make_step_inputs(wl)
    ids = np.arange(V)
    out = (ids // (V // 10) == 3) if mask.startswith("a tenth") else (np.random.default_rng(V).random(V) < 0.5)
    for arr in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond):
        arr[:, :, out] = wk._store(np.full(1, -np.inf, np.float32), dtype)[0]
    prev = oracle_prime(inp)
    rep, got, ref = check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
    assert not np.any(got.status & 16)


# rows that one CTA does not hold: clusters of two, four and eight with ragged last segments, and more rows than there is
# room for their clusters (which the kernel for many rows takes)
@pytest.mark.parametrize("V,K,dtype,B,W", [(40008, 300, wk.F32, 1, 3), (65528, 700, wk.F16, 2, 5), (65544, 300, wk.F32, 1, 4), (65536, 500, wk.F32, 4, 9),
                                           (131080, 2000, wk.BF16, 1, 3), (262152, 1500, wk.F16, 1, 2), (262144, 500, wk.BF16, 2, 5),
                                           (300008, 100, wk.F32, 1, 1)])
def test_rows_shared_by_a_cluster(V, K, dtype, B, W):
    _check(f"cluster{V}", B=B, W=W, V=V, dtype=dtype, top_k=K, seed=V % 1000)


@pytest.mark.parametrize("V,K,dtype,B,W,temperature", [(8192, 300, wk.BF16, 3, 60, 1.0), (65536, 2000, wk.BF16, 3, 60, 1.0),
                                                       (65536, 500, wk.F32, 6, 30, 0.9), (50264, 100, wk.F16, 4, 50, 1.0)])
def test_a_sequence_alone_gives_the_same_bits(V, K, dtype, B, W, temperature):
    # one sequence's rows by clusters, the same rows in a batch by the kernel for many rows
    from gpu_harness import gpu_step, oracle_prime, step_kwargs
    import oracle
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, temperature=temperature, seed=V % 77)
    inp = wk.make_step_inputs(wl)
    prev = oracle_prime(inp)
    batch = gpu_step(inp.cond, inp.uncond, prev.tokens, prev.probs, **step_kwargs(inp))
    one = lambda a: None if a is None else np.ascontiguousarray(a[:1])
    q = oracle.Probs(one(prev.probs.tok_prob), one(prev.probs.ids), one(prev.probs.vals), one(prev.probs.cnt))
    kw = step_kwargs(inp, win_len=one(inp.win_len), pos_base=one(inp.pos_base))
    alone = gpu_step(one(inp.cond), one(inp.uncond), one(prev.tokens), q, **kw)
    for name in ("accept_len", "tokens", "tok_prob", "ids", "vals", "cnt", "flags", "status"):
        assert getattr(alone, name).tobytes() == getattr(batch, name)[:1].tobytes(), name


# One CTA per row, clusters of two and four, many rows; more candidates than the lists hold and fewer; blocks at the row's ends;
# several rows to a CTA, some of them ordinary.
@pytest.mark.parametrize("V,K,dtype,B,W", [(16384, 500, wk.BF16, 1, 3), (65536, 2000, wk.BF16, 1, 4), (65536, 300, wk.F32, 1, 3),
                                           (65536, 100, wk.F16, 2, 77), (65536, 2000, wk.BF16, 2, 80), (5000, 300, wk.BF16, 3, 110),
                                           (16384, 1000, wk.F32, 2, 90), (50264, 5000, wk.F16, 2, 75), (2056, 64, wk.F32, 4, 100)])
@pytest.mark.parametrize("where", ["start", "middle", "end"])
def test_top_k_in_one_block_of_ids(V, K, dtype, B, W, where):
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, seed=V + W, peaks=0)
    inp = wk.make_step_inputs(wl)
    n = max(V // 8, K + K // 2)
    begin = {"start": 0, "middle": (V - n) // 3, "end": V - n}[where]
    for arr in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond):
        f = wk._as_f32(arr, dtype).copy()
        f[:, : W - W // 3, begin:begin + n] += 12.0  # (the last third of the rows is ordinary)
        arr[:] = wk._store(f, dtype)
    prev = oracle_prime(inp)
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)


@pytest.mark.parametrize("lowest", [-np.inf, -65504.0])
@pytest.mark.parametrize("V,K,dtype,B,W,left", [(16384, 500, wk.BF16, 1, 3, 2048), (65536, 2000, wk.BF16, 1, 4, 8192), (65536, 2000, wk.BF16, 2, 80, 8192),
                                                (65536, 100, wk.F16, 2, 77, 8192), (50264, 500, wk.BF16, 2, 75, 6000), (16384, 1000, wk.F32, 2, 90, 1500),
                                                (8192, 300, wk.F32, 2, 90, 290)])
def test_all_but_a_block_masked(V, K, dtype, B, W, left, lowest):
    # image tokens only: fewer of the sample's groups are unmasked than the threshold's rank; the last shape has fewer tokens than K left
    from gpu_harness import check_parity, oracle_prime, step_kwargs
    wl = wk.CONFIGS["cfg2"].scaled(B=B, W=W, V=V, dtype=dtype, top_k=K, seed=V + W, peaks=0)
    inp = wk.make_step_inputs(wl)
    out = np.ones(V, bool)
    out[V // 5:V // 5 + left] = False
    for arr in (inp.cond, inp.uncond, inp.prev_cond, inp.prev_uncond):
        arr[:, :, out] = wk._store(np.full(1, lowest, np.float32), dtype)[0]
    prev = oracle_prime(inp)
    check_parity(inp.cond, inp.uncond, prev.tokens, prev.probs, step_kwargs(inp), inp.win_len)
