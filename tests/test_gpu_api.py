"""GPU tests of the C ABI's argument checking and edge cases (host-side failures only)."""
import numpy as np
import pytest

from workloads import SHAPES, ModelShape, make_prompt, make_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    from paper_2304_04487_b200 import Engine
    shape = SHAPES["tiny-fp32"]
    w = make_weights(shape, seed=0)
    return Engine, shape, w


def test_argument_errors_leave_engine_usable(setup):
    from paper_2304_04487_b200 import LlmaError
    Engine, shape, w = setup
    eng = Engine(shape, w, max_seq=48, max_ref=16, max_k=4)
    with pytest.raises(LlmaError) as ei:
        eng.llma_step(1, 2)                              # nothing prefilled
    assert ei.value.status == -6
    prompt = make_prompt(20, shape.vocab, seed=1)
    for bad, code in ((list(prompt[:5]) + [shape.vocab], -3), ([-1], -3), (list(range(49)), -4), ([], -9)):
        with pytest.raises(LlmaError) as ei:
            eng.llma_prefill(0, bad)
        assert ei.value.status == code
    with pytest.raises(LlmaError) as ei:
        eng.llma_prefill(1, prompt)                      # only one slot
    assert ei.value.status == -4
    eng.llma_prefill(0, prompt)
    for (n, k) in ((0, 2), (1, 5), (1, -1)):
        with pytest.raises(LlmaError) as ei:
            eng.llma_step(n, k)
        assert ei.value.status == -9
    with pytest.raises(LlmaError) as ei:
        eng.llma_set_reference(0, list(range(17)))
    assert ei.value.status == -5
    with pytest.raises(LlmaError) as ei:
        eng.llma_set_reference(0, [1, 2, 3, 4], [0, 3, 2, 4])
    assert ei.value.status == -5
    with pytest.raises(LlmaError) as ei:
        eng.llma_set_reference(0, [1, 2, shape.vocab])
    assert ei.value.status == -3
    with pytest.raises(LlmaError) as ei:
        eng.llma_generate(30, 1, 2)                      # 19 cached + 30 > 48
    assert ei.value.status == -4
    with pytest.raises(LlmaError) as ei:
        eng.llma_debug_logits()                          # keep_logits was not requested
    assert ei.value.status == -6
    (toks,), st = eng.llma_generate(29, 1, 2)            # exactly fills the cache
    assert len(toks) == 29 and eng.llma_kv_len(0) == 48
    with pytest.raises(LlmaError) as ei:
        eng.llma_step(1, 2)                              # cache is full
    assert ei.value.status == -4
    eng.llma_rewind(0)
    (again,), _ = eng.llma_generate(29, 1, 0)
    assert again == toks
    eng.llma_reset(0)
    with pytest.raises(LlmaError):
        eng.llma_kv_len(0)


def test_unsupported_configs_rejected(setup):
    from paper_2304_04487_b200 import LlmaError
    Engine, shape, w = setup
    with pytest.raises(LlmaError) as ei:
        Engine(shape, w, max_seq=32, max_ref=8, max_k=16, max_batch=16)  # 16 * 17 rows > 256
    assert ei.value.status == -2
    with pytest.raises(LlmaError) as ei:
        Engine(shape, w, max_seq=32, max_ref=8, max_k=2, gemm_impl=2)    # tensor-core GEMM needs bf16
    assert ei.value.status == -2


def test_edge_cases(setup):
    Engine, shape, w = setup
    eng = Engine(shape, w, max_seq=64, max_ref=32, max_k=8, eos_id=-1)
    # one-token prompt: nothing to cache, first step runs at position 0
    eng.llma_prefill(0, [5])
    assert eng.llma_kv_len(0) == 0
    (g,), st = eng.llma_generate(20, 1, 0)
    assert len(g) == 20
    # zero new tokens is a no-op
    (z,), st0 = eng.llma_generate(0, 1, 4)
    assert z == [] and st0.steps == 0
    # a match right at the end of a document copies nothing; a copy longer than what is left to
    # emit is cut so that exactly max_new tokens come out
    eng.llma_set_reference(0, g[:6] + g[10:14], [0, 6, 10])
    eng.llma_rewind(0)
    (t,), st = eng.llma_generate(7, 1, 8)
    assert t == g[:7] and st.tokens == 7
    eng.llma_rewind(0)
    (t,), st = eng.llma_generate(20, 1, 8)
    assert t == g
    # EOS: generation stops right after the first occurrence of eos_id
    eos = g[9]
    first = g.index(eos)
    e2 = Engine(shape, w, max_seq=64, max_ref=32, max_k=8, eos_id=eos)
    e2.llma_prefill(0, [5])
    e2.llma_set_reference(0, g[:20])
    (t,), st = e2.llma_generate(20, 1, 8)
    assert t == g[:first + 1]


def test_microbench_mma_runs_and_rejects_bad_arguments():
    """The tensor-core timing probe: a plausible figure for a legal shape, LLMA_ERR_ARG for the rest."""
    from paper_2304_04487_b200 import LlmaError, llma_microbench_mma
    t32 = llma_microbench_mma(32, 1, 256, 0)
    t256 = llma_microbench_mma(256, 2, 256, 1)
    assert 10.0 < t32 < 1000.0 and 10.0 < t256 < 1000.0, (t32, t256)
    for bad in ((24, 1, 256, 0), (272, 1, 256, 0), (256, 3, 256, 0), (32, 1, 0, 0), (32, 1, 256, 5), (0, 1, 1, 0)):
        with pytest.raises(LlmaError):
            llma_microbench_mma(*bad)


# shapes whose steps are launched kernel by kernel: tensor cores on request, and CUDA cores where two rows fit a pass
LAUNCHED = {"tiny-bf16": (SHAPES["tiny-bf16"], 2), "fp32-launched": (ModelShape("fp32-launched", 2, 128, 2, 64, 8192, 515, "fp32"), 0)}


@pytest.mark.parametrize("name,launched", [("tiny-fp32", False), ("tiny-bf16", False), ("tiny-bf16", True), ("fp32-launched", True)])
def test_engine_on_the_default_stream(setup, name, launched):
    """cuda_stream = NULL: CUDA does not capture the legacy default stream, so every entry point has to do without graphs.
    Same tokens as on a stream of its own, whether a step is launched directly or replayed."""
    import torch
    Engine = setup[0]
    shape, impl = LAUNCHED[name] if launched else (SHAPES[name], 0)
    w = make_weights(shape, seed=0)
    prompt = make_prompt(20, shape.vocab, seed=1)
    own = Engine(shape, w, max_seq=96, max_ref=64, max_k=4, gemm_impl=impl)
    null = Engine(shape, w, max_seq=96, max_ref=64, max_k=4, gemm_impl=impl, stream=torch.cuda.default_stream())
    assert null.stream.cuda_stream == 0
    out = []
    for eng in (own, null):
        eng.llma_prefill(0, prompt)
        (y,), st = eng.llma_generate(24, 1, 0)
        assert (st.launches > 24) == launched
        eng.llma_set_reference(0, y)
        for _ in range(5):                     # 25 steps: launched directly, captured, replayed
            steps = []
            eng.llma_rewind(0)
            for _ in range(5):
                steps += eng.llma_step(1, 4)[0]
            assert steps == y[:len(steps)]
        eng.llma_rewind(0)
        (z,), sz = eng.llma_generate(24, 1, 4)
        eng.llma_rewind(0)
        sf = eng.llma_generate_forced(0, [(3, 2)] * 6, y[:12])
        out.append((y, steps, z, st.steps, st.launches, sz.steps, sz.launches, sf.tokens, sf.launches))
    assert out[0] == out[1]
    assert out[0][2] == out[0][0] and out[0][1] == out[0][0][:len(out[0][1])]


@pytest.mark.parametrize("name", ["tiny-fp32", *LAUNCHED])   # whole steps, which make no graphs; launches
def test_more_step_shapes_than_graphs_are_kept(setup, name):
    """Captured steps are kept for the last 64 (n, k); one that has made room for another is captured again."""
    Engine, shape, w = setup
    impl = 0
    if name in LAUNCHED:
        shape, impl = LAUNCHED[name]
        w = make_weights(shape, seed=0)
    eng = Engine(shape, w, max_seq=64, max_ref=32, max_k=4, gemm_impl=impl)
    eng.llma_prefill(0, make_prompt(20, shape.vocab, seed=1))
    (y,), st = eng.llma_generate(12, 1, 0)
    assert (st.launches > 12) == (name in LAUNCHED)
    eng.llma_set_reference(0, y)
    for turn in range(3):
        for n in range(1, 71):
            eng.llma_rewind(0)
            got = []
            while len(got) < 6:
                got += eng.llma_step(n, 4)[0]
            assert got[:6] == y[:6], (turn, n)
        for n in range(1, 71):
            eng.llma_rewind(0)
            (z,), _ = eng.llma_generate(6, n, 4)
            assert z == y[:6], (turn, n)


class _OnDevice:
    """Device tensors in the form in which one engine lends its weights to another."""

    def __init__(self, dev):
        self._dev = dev


def _shifted(t, values=1):
    """The same values `values` elements past a 256-byte boundary."""
    import torch
    flat = torch.empty(t.numel() + values, dtype=t.dtype, device=t.device)
    flat[values:] = t.flatten()
    return flat[values:].view(t.shape)


@pytest.mark.parametrize("name,B,k,P", [("tiny-fp32", 1, 4, 40),      # CUDA cores
                                        ("small-bf16", 1, 4, 200),    # prompt kernels, up to 16 rows
                                        ("small-bf16", 5, 7, 100)])   # 33 to 256 rows
def test_gains_and_embeddings_need_no_alignment(name, B, k, P):
    """Norm gains and the embedding table may be views into larger buffers at any element: same bits as on a boundary."""
    from paper_2304_04487_b200 import Engine
    shape = SHAPES[name]
    w = make_weights(shape, seed=0)
    rng = np.random.default_rng(5)
    for n in w:
        if w[n].ndim == 1:
            w[n] = rng.uniform(0.5, 1.5, w[n].shape).astype(np.float32)   # gains that differ from one another
    a = Engine(shape, w, max_seq=P + 40, max_ref=32, max_k=k, max_batch=B, keep_logits=True)
    dev = {n: _shifted(t) if t.ndim == 1 or n == "tok_emb" else t for n, t in a._dev.items()}
    assert all(dev[n].data_ptr() % 16 for n in dev if dev[n].ndim == 1 or n == "tok_emb")
    b = Engine(shape, None, max_seq=P + 40, max_ref=32, max_k=k, max_batch=B, keep_logits=True, share_weights_with=_OnDevice(dev))
    out = []
    for eng in (a, b):
        for s in range(B):
            eng.llma_prefill(s, make_prompt(P + s, shape.vocab, seed=s))
            eng.llma_set_reference(s, make_prompt(P + s, shape.vocab, seed=s)[:32])
        rows = []
        for _ in range(4):
            toks = eng.llma_step(1, k)
            logits = eng.llma_debug_logits()
            rows.append((toks, [logits[s * (k + 1):s * (k + 1) + i.k_eff + 1].copy() for s, i in enumerate(eng.llma_last_step_info())]))
        out.append(rows)
    for (ta, la), (tb, lb) in zip(*out):
        assert ta == tb
        assert all(np.array_equal(x, y) for x, y in zip(la, lb))


@pytest.mark.parametrize("name", ["tiny-fp32", "tiny-bf16"])
def test_misaligned_matrices_are_rejected(name):
    from paper_2304_04487_b200 import Engine, LlmaError
    shape = SHAPES[name]
    a = Engine(shape, make_weights(shape, seed=0), max_seq=32, max_ref=8, max_k=2)
    for n in ("wq.0", "wo.1", "w_up.0", "w_down.1", "lm_head"):
        for impl in ((1,) if name == "tiny-fp32" else (1, 2)):
            with pytest.raises(LlmaError) as ei:
                Engine(shape, None, max_seq=32, max_ref=8, max_k=2, gemm_impl=impl,
                       share_weights_with=_OnDevice({**a._dev, n: _shifted(a._dev[n])}))
            assert ei.value.status == -2


def test_prompt_passes_shrink_where_memory_is_short():
    """An engine whose full-sized prompt buffers do not fit takes smaller passes instead of failing: the same K/V rows.  (In a process
    of its own, which takes all but part of the memory that the engine would like to have.)"""
    import os
    import subprocess
    import sys
    code = """
import numpy as np, torch
from paper_2304_04487_b200 import Engine
from workloads import ModelShape, make_prompt, make_weights
shape = ModelShape("wide-ffn", 1, 1024, 8, 128, 16384, 1000, "bf16")
kw = dict(max_seq=2081, max_ref=8, max_k=1)
a = Engine(shape, make_weights(shape, seed=0), **kw)
prompt = make_prompt(2049, shape.vocab, seed=3)
free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]
at = (0, 127, 128, 1023, 1024, 2047)
def rows(eng):
    eng.llma_prefill(0, prompt)
    return [eng.llma_debug_kv_row(0, 0, p, which) for p in at for which in (0, 1)] + eng.llma_generate(4, 1, 0)[0]
want = rows(a)
before = free()
b = Engine(shape, None, share_weights_with=a, **kw)
size = before - free()
b.llma_destroy()
assert size > 168 << 20                       # 2048 positions of 82 KB, and the rest
taken = torch.empty(free() - (size - (100 << 20)), dtype=torch.uint8, device="cuda")
before = free()
c = Engine(shape, None, share_weights_with=a, **kw)
assert before - free() <= size - (80 << 20)
assert all(np.array_equal(x, y) for x, y in zip(rows(c), want))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)


def test_whole_steps_do_without_where_memory_is_short():
    """An engine for whose whole steps there is no room launches its steps kernel by kernel instead of failing: the same tokens.  (In a
    process of its own, which takes all but part of the memory that the engine would like to have.)"""
    import os
    import subprocess
    import sys
    code = """
import torch
from paper_2304_04487_b200 import Engine
from workloads import ModelShape, make_prompt, make_weights
shape = ModelShape("words", 1, 1024, 8, 128, 2048, 300, "fp32")
kw = dict(max_seq=40, max_ref=8, max_k=7, max_batch=32)                 # 256 rows: 16 MB of words
a = Engine(shape, make_weights(shape, seed=0), **kw)
prompt = make_prompt(9, shape.vocab, seed=3)
free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]
def decode(eng):
    eng.llma_prefill(0, prompt)
    (y,), st = (lambda t, s: (t[:1], s))(*eng.llma_generate(6, 1, 0))
    return y, st.launches
want, launches = decode(a)
assert launches == 1
before = free()
b = Engine(shape, None, share_weights_with=a, **kw)
size = before - free()
b.llma_destroy()
taken = torch.empty(free() - (size - (8 << 20)), dtype=torch.uint8, device="cuda")
c = Engine(shape, None, share_weights_with=a, **kw)
got, launches = decode(c)
assert got == want and launches > 6
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)
