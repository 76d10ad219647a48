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
