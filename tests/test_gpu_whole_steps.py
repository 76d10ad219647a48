"""Decoding steps that run whole in one launch: many steps per launch, launches that end early or follow one another, and
more rows than one pass over the weights takes.  The step itself is compared with the oracle in test_gpu_parity.py."""
import numpy as np
import pytest

from workloads import ModelShape, make_prompt, make_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,hd,ffn,vocab,k,B,N", [
    (64, 1, 64, 64, 77, 3, 1, 33),          # fewer units than SMs everywhere; one step more than a launch takes
    (192, 3, 64, 320, 1001, 6, 3, 70),      # 21 rows: two passes; odd vocabulary, units that end inside it
    (512, 4, 128, 1408, 5000, 2, 1, 96)])   # long units: pieces that the warps request themselves
def test_generate_equals_single_steps(d, heads, hd, ffn, vocab, k, B, N):
    from paper_2304_04487_b200 import Engine
    shape = ModelShape(f"whole-{d}", 2, d, heads, hd, ffn, vocab, "fp32")
    eng = Engine(shape, make_weights(shape, seed=0, std=0.05), max_seq=20 + N + k + 8, max_ref=N, max_k=k, max_batch=B, keep_logits=True)
    for s in range(B):
        eng.llma_prefill(s, make_prompt(20 - s, vocab, seed=40 + s))
    greedy, st = eng.llma_generate(N, 1, 0)
    assert st.steps == B * N and all(len(y) == N for y in greedy)
    eng.llma_step(1, 0)
    want = eng.llma_debug_logits().reshape(B, k + 1, vocab)[:, 0]
    for s in range(B):
        eng.llma_set_reference(s, greedy[s][:N // 2] + greedy[s][N // 3:][:N // 2])
    for turn in range(2):
        for s in range(B):
            eng.llma_rewind(s)
        toks, st = eng.llma_generate(N, 1, k)
        assert toks == greedy and st.steps < B * N and st.copied_accepted > 0
        eng.llma_step(1, 0)                 # the position after the last: every cache row of the run is read
        assert np.array_equal(eng.llma_debug_logits().reshape(B, k + 1, vocab)[:, 0], want)
    for s in range(B):
        eng.llma_rewind(s)
    got = [[] for _ in range(B)]
    while min(map(len, got)) < N:
        for s, t in enumerate(eng.llma_step(1, k)):
            got[s] += t
    assert [g[:N] for g in got] == greedy
    eng.llma_destroy()


@pytest.mark.parametrize("impl", [0, 2])   # whole steps (narrow, few rows, short contexts), and the launches that they stand in for
@pytest.mark.parametrize("name,k", [("tiny-bf16", 8), ("small-bf16", 15)])
def test_narrow_decoders_both_ways(name, k, impl):
    from oracle import model as OM
    from parity import step_parity
    from paper_2304_04487_b200 import Engine
    from workloads import SHAPES, build_reference
    shape = SHAPES[name]
    w = make_weights(shape, seed=0)
    P, N = 290, 24
    prompt = make_prompt(P, shape.vocab, seed=2)
    eng = Engine(shape, w, max_seq=P + N + 40, max_ref=200, max_k=k, gemm_impl=impl, keep_logits=True)
    assert eng.llma_gemm_impl() == 2
    eng.llma_prefill(0, prompt)
    (y,), st = eng.llma_generate(N, 1, 0)
    assert st.launches == (1 if impl == 0 else 1 + N * (3 + 6 * shape.n_layers))
    ref, offs, _ = build_reference(y, [60, 60, 40], 0.7, shape.vocab, seed=1)
    rep = step_parity(eng, OM.OracleModel(shape, w, max_seq=P + N + 40), prompt, ref, offs, 1, k, N, "bf16")
    assert rep.max_logit_err <= 2e-2 and rep.near_ties <= 3 and rep.trigger_steps > 0
    prof = eng.llma_profile_steps(1, k, 2)                  # launch by launch, on the same engine
    assert prof["_total"]["launches_per_step"] == 4 + 5 * shape.n_layers   # (the two attention kernels count as one)
    eng.llma_destroy()


def test_passes_change_from_step_to_step():
    """Steps of one, two and three passes over the weights in turn, in one launch: the weights that are on their way into a step's ring
    are those of its own passes."""
    from paper_2304_04487_b200 import Engine
    B, k, N = 4, 9, 120                       # 4 to 40 rows
    shape = ModelShape("passes", 2, 128, 2, 64, 384, 515, "fp32")
    eng = Engine(shape, make_weights(shape, seed=0, std=0.05), max_seq=40 + N, max_ref=2 * N, max_k=k, max_batch=B, keep_logits=True)
    for s in range(B):
        eng.llma_prefill(s, make_prompt(20 + s, shape.vocab, seed=70 + s))
    rng = np.random.default_rng(3)
    y = [int(t) for t in rng.integers(0, shape.vocab, N)]
    eng.llma_generate_forced(-1, [(1, 1)] * N, y)   # four rows a step
    eng.llma_step(1, 0)
    want = eng.llma_debug_logits().reshape(B, k + 1, -1)[:, 0]
    for turn in range(20):
        for s in range(B):
            eng.llma_rewind(s)
        trace, left = [], N
        while left:
            rows = int(rng.choice([1, 4, 5, 8, 9, 10]))
            out = min(left, int(rng.integers(1, rows + 1)))
            trace.append((rows, out))
            left -= out
        st = eng.llma_generate_forced(-1, trace, y)
        assert st.steps == B * len(trace)
        eng.llma_step(1, 0)
        assert np.array_equal(eng.llma_debug_logits().reshape(B, k + 1, -1)[:, 0], want)
    eng.llma_destroy()


@pytest.mark.parametrize("name", ["tiny-bf16", "tiny-fp32"])
def test_launches_that_give_up_are_repeated(name):
    """A launch of whole steps whose CTAs did not get onto the GPU together leaves its mark in the error word: launches behind it do
    nothing, the call launches them again and gives what it gives undisturbed.  (The mark is preset; no wait is made to run out.)"""
    from paper_2304_04487_b200 import Engine
    from workloads import SHAPES
    shape = SHAPES[name]
    N, k = 70, 4                                                   # more than two launches
    eng = Engine(shape, make_weights(shape, seed=0), max_seq=30 + N + k, max_ref=N, max_k=k)
    eng.llma_prefill(0, make_prompt(20, shape.vocab, seed=1))
    (y,), st = eng.llma_generate(N, 1, 0)
    assert st.launches == 3
    eng.llma_set_reference(0, y)

    def generate(k):
        (toks,), st = eng.llma_generate(N, 1, k)
        assert toks == y and st.tokens == N and st.steps == N - st.copied_accepted
        return st.launches

    def steps():
        got = []
        while len(got) < N:
            eng.llma_debug_set_device_error(4)
            got += eng.llma_step(1, k)[0]
        assert got[:N] == y

    def replay(trace):
        st = eng.llma_generate_forced(0, trace, y)
        assert (st.steps, st.tokens) == (len(trace), N)

    for call in (lambda: generate(0), lambda: generate(k), steps, lambda: replay([(1, 1)] * 10 + [(5, 3)] * 20)):
        eng.llma_rewind(0)
        eng.llma_debug_set_device_error(4)
        call()
    eng.llma_rewind(0)
    eng.llma_debug_set_device_error(4)
    assert generate(0) > 3                                         # those that did nothing, and those that did
    eng.llma_destroy()


def test_positions_without_weight_come_first():
    """Scores of minus infinity (products that overflow) at the first positions, where a warp of the attention has seen nothing else yet:
    they weigh nothing, as they do for the oracle."""
    from oracle import model as OM
    from parity import step_parity
    from paper_2304_04487_b200 import Engine
    V, d, bad = 77, 64, 8
    shape = ModelShape("overflow", 1, d, 1, 64, 64, V, "fp32")
    w = make_weights(shape, seed=0, std=0.3)
    w["tok_emb"][:, :2] = [1.0, 0.0]          # ordinary tokens: a query of 1e20 in a slow rotary pair, a key of 0
    w["tok_emb"][:bad, :2] = [0.0, -1.0]      # the others: a query of 0, a key of -1e20
    w["lm_head"][:bad] = 0.0
    for name, col in (("wq.0", 0), ("wk.0", 1)):
        w[name][31], w[name][63] = 0.0, 0.0
        w[name][31, col] = 1e20
    prompt = list(range(bad)) + [int(t) for t in make_prompt(7, V - bad, seed=1) + bad]
    eng = Engine(shape, w, max_seq=64, max_ref=32, max_k=3, keep_logits=True)
    rep = step_parity(eng, OM.OracleModel(shape, w, max_seq=64), prompt, prompt[bad:], None, 1, 3, 20, "fp32")
    assert np.isfinite(rep.max_logit_scale) and min(rep.tokens) >= bad and rep.near_ties == 0
    eng.llma_destroy()


@pytest.mark.parametrize("whole,d,heads,hd,ffn,vocab,dtype,k,B,max_seq", [
    (True, 256, 4, 64, 1024, 515, "fp32", 18, 4, 96),        # 76 rows: five passes either way
    (True, 320, 5, 64, 4096, 301, "fp32", 15, 1, 96),        # 16 rows: three passes of six, the launches two of eight
    (False, 320, 5, 64, 8192, 301, "fp32", 4, 1, 96),        # two rows a pass
    (False, 320, 5, 64, 4096, 301, "fp32", 8, 4, 96),        # 36 rows: six passes for three
    (True, 320, 5, 64, 8192, 301, "fp32", 1, 1, 96),         # two rows, one pass
    (True, 512, 8, 64, 2048, 301, "bf16", 15, 1, 96), (False, 512, 8, 64, 2048, 301, "bf16", 15, 1, 768),   # the line of positions
    (True, 512, 8, 64, 2048, 301, "bf16", 7, 1, 768), (False, 512, 8, 64, 2048, 301, "bf16", 7, 1, 769),
    (False, 512, 8, 64, 4096, 301, "bf16", 8, 1, 96), (True, 512, 8, 64, 4096, 301, "bf16", 4, 1, 96),      # more than a pass; one
    (False, 512, 4, 64, 512, 60000, "bf16", 15, 1, 600), (True, 512, 4, 64, 512, 60000, "bf16", 7, 1, 600)])  # the LM head's share
def test_whole_steps_where_they_pay(whole, d, heads, hd, ffn, vocab, dtype, k, B, max_seq):
    from paper_2304_04487_b200 import Engine
    shape = ModelShape(f"pay-{d}-{ffn}", 1, d, heads, hd, ffn, vocab, dtype)
    eng = Engine(shape, make_weights(shape, seed=0, std=0.05), max_seq=max_seq, max_ref=64, max_k=k, max_batch=B)
    for s in range(B):
        eng.llma_prefill(s, make_prompt(20 + s, vocab, seed=s))
    greedy, st = eng.llma_generate(20, 1, 0)
    assert (st.launches == 1) == whole
    for s in range(B):
        eng.llma_set_reference(s, greedy[s])
        eng.llma_rewind(s)
    assert eng.llma_generate(20, 1, k)[0] == greedy
    eng.llma_destroy()
