"""llma_generate with an EOS token: steps are launched in batches, so those after the last sequence has ended run without rows."""
import pytest

from workloads import SHAPES, make_prompt, make_weights

pytestmark = pytest.mark.gpu

N, K = 40, 8


def _engine(name, B, max_k, impl, eos=-1, share=None):
    from paper_2304_04487_b200 import Engine
    shape = SHAPES[name]
    return Engine(shape, None if share else make_weights(shape, seed=0), max_seq=100 + N, max_ref=N, max_k=max_k, max_batch=B,
                  gemm_impl=impl, eos_id=eos, share_weights_with=share)


def _fresh(tokens, most):
    """The last of the first `most` tokens that has not occurred before."""
    return [t for i, t in enumerate(tokens[:most]) if t not in tokens[:i]][-1]


@pytest.mark.parametrize("name,B,max_k,impl", [
    ("tiny-bf16", 1, 8, 2), ("tiny-bf16", 2, 7, 2),      # tensor-core launches of up to 16 rows
    ("small-bf16", 1, 20, 2), ("small-bf16", 3, 8, 2),   # ... 32 rows
    ("small-bf16", 5, 8, 2),                             # ... more: the wide kernel
    ("mid-bf16", 1, 8, 0), ("mid-bf16", 3, 8, 0),        # what the automatic choice takes at width 1024
    ("tiny-bf16", 1, 8, 0), ("tiny-bf16", 2, 7, 0),      # whole steps
    ("tiny-fp32", 1, 8, 0), ("tiny-fp32", 3, 8, 0)])
def test_generate_stops_at_eos(name, B, max_k, impl):
    shape = SHAPES[name]
    k = min(K, max_k)
    plain = _engine(name, B, max_k, impl)
    head = make_prompt(24, shape.vocab, seed=3)
    plain.llma_prefill(0, head)
    lead = plain.llma_generate(12, 1, 0)[0][0]
    # all sequences on the same text, each a token further: they all end, one after the other.  Then texts of their own: one ends
    together = [list(head) + lead[:s] for s in range(B)]
    apart = [make_prompt(24 + 3 * s, shape.vocab, seed=3 + s) for s in range(B)]
    for prompts in (together, apart):
        for s, p in enumerate(prompts):
            plain.llma_prefill(s, p)
        full, _ = plain.llma_generate(N, 1, 0)
        eos = _fresh(full[0], 10)
        want = [y[:y.index(eos) + 1] if eos in y else y for y in full]
        assert len(want[0]) <= 10 and (prompts is apart or all(len(w) < N for w in want))
        eng = _engine(name, B, max_k, impl, eos, plain)
        for s, p in enumerate(prompts):
            eng.llma_prefill(s, p)
            eng.llma_set_reference(s, full[s])
        for copy in (0, k, 0):
            got, st = eng.llma_generate(N, 1, copy)
            assert got == want and st.tokens == sum(map(len, want))
            for s in range(B):
                eng.llma_rewind(s)
        eng.llma_destroy()
    plain.llma_destroy()
