"""Engines of both kinds side by side, each with a thread and a stream of its own: every call gives what it gives alone."""
import threading
import time

import pytest

from workloads import SHAPES, build_reference, make_prompt, make_weights

pytestmark = pytest.mark.gpu


def _engine(name, k, impl=0):
    from paper_2304_04487_b200 import Engine
    shape = SHAPES[name]
    eng = Engine(shape, make_weights(shape, seed=0), max_seq=220, max_ref=128, max_k=k, gemm_impl=impl)
    eng.llma_prefill(0, make_prompt(100, shape.vocab, seed=1))
    (y,), _ = eng.llma_generate(48, 1, 0)
    ref, offs, _ = build_reference(y, [128], 0.7, shape.vocab, seed=0)
    eng.llma_set_reference(0, ref, offs)
    return eng, y


def _generate(eng, y, k):
    eng.llma_rewind(0)
    (toks,), _ = eng.llma_generate(48, 1, k)
    assert toks == y


def _step(eng, y, k):
    eng.llma_rewind(0)
    got = []
    while len(got) < 48:
        got += eng.llma_step(1, k)[0]
    assert got[:48] == y


def _replay(eng, y, k):
    eng.llma_rewind(0)
    assert eng.llma_generate_forced(0, [(1, 1)] * 24 + [(3, 2)] * 12, y).tokens == 48
    eng.llma_rewind(0)
    eng.llma_profile_steps(1, k, 3)


def _product(noalloc):
    import torch
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16, llma_gemm_rows32_bf16_noalloc
    gemm = llma_gemm_rows32_bf16_noalloc if noalloc else llma_gemm_rows32_bf16
    g = torch.Generator(device="cuda").manual_seed(2)
    W = (torch.randn(4096, 4096, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    a = torch.randn(32, 4096, device="cuda", generator=g).to(torch.bfloat16)
    want, out, st = torch.empty(32, 4096, device="cuda"), torch.empty(32, 4096, device="cuda"), torch.cuda.Stream()
    gemm(W, a, want)
    torch.cuda.synchronize()

    def work():
        gemm(W, a, out, stream=st)
        with torch.cuda.stream(st):
            assert torch.equal(out, want)
    return work


def _side_by_side(jobs, seconds):
    """Every job again and again in a thread of its own, for some time."""
    failed, done, until = [], [0] * len(jobs), time.monotonic() + seconds

    def loop(i):
        try:
            while time.monotonic() < until and not failed:
                jobs[i]()
                done[i] += 1
        except Exception as e:  # noqa: BLE001 (a thread's failure is the test's)
            failed.append((i, e))

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed and min(done) > 0, (failed, done)


@pytest.mark.parametrize("whole,tiles", [("tiny-fp32", "mid-bf16"), ("small-bf16", "mid-bf16"), ("tiny-bf16", "llama7b-1layer")])
def test_whole_steps_beside_other_engines(whole, tiles):
    a, ya = _engine(whole, 4)
    b, yb = _engine(whole, 4)
    c, yc = _engine(tiles, 8)
    jobs = [lambda: (_generate(a, ya, 4), _replay(a, ya, 4)), lambda: (_step(b, yb, 4), _generate(b, yb, 4)),
            lambda: (_generate(c, yc, 8), _step(c, yc, 8), _replay(c, yc, 8)), _product(False), _product(True)]
    _side_by_side(jobs, 1.0)
    for e in (a, b, c):
        e.llma_destroy()


def test_engines_come_and_go_beside_others():
    """Engines of both kinds are made, used and destroyed while others decode: what a new engine launches takes turns from its first
    launch on, the one that its creation makes included."""
    import torch
    from paper_2304_04487_b200 import Engine
    old, y = _engine("mid-bf16", 8)
    names = ("tiny-fp32", "mid-bf16", "tiny-bf16")
    weights = {n: make_weights(SHAPES[n], seed=0) for n in names}
    streams = {n: torch.cuda.Stream() for n in names}       # (streams of torch's pool come round again)
    want = {}

    def make():
        for n in names:
            eng = Engine(SHAPES[n], weights[n], max_seq=120, max_ref=16, max_k=2, stream=streams[n])
            eng.llma_prefill(0, make_prompt(50, SHAPES[n].vocab, seed=9))
            (toks,), _ = eng.llma_generate(20, 1, 0)
            assert want.setdefault(n, toks) == toks
            eng.llma_destroy()
    make()
    _side_by_side([make, lambda: (_generate(old, y, 8), _replay(old, y, 8)), _product(False)], 2.0)
    old.llma_destroy()


def test_stream_that_has_part_of_the_sms():
    """An engine on a stream of a green context, which has 64 SMs: a launch that needs every SM is refused there, so steps are launched
    kernel by kernel.  The same tokens."""
    import torch
    driver = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert r[0] == driver.CUresult.CUDA_SUCCESS, r
        return r[1] if len(r) == 2 else r[1:]
    torch.zeros(1, device="cuda")
    dev = ok(driver.cuDeviceGet(0))
    sms = ok(driver.cuDeviceGetDevResource(dev, driver.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(driver.cuDevSmResourceSplitByCount(1, sms, 0, 64))
    green = ok(driver.cuGreenCtxCreate(ok(driver.cuDevResourceGenerateDesc([groups[0]], 1)), dev, driver.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    part = torch.cuda.ExternalStream(int(ok(driver.cuGreenCtxStreamCreate(green, driver.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))))
    from paper_2304_04487_b200 import Engine
    shape = SHAPES["tiny-fp32"]
    w = make_weights(shape, seed=0)
    got = []
    for stream in (None, part):
        eng = Engine(shape, w, max_seq=96, max_ref=64, max_k=4, stream=stream)
        eng.llma_prefill(0, make_prompt(20, shape.vocab, seed=1))
        (y,), st = eng.llma_generate(24, 1, 0)
        eng.llma_set_reference(0, y)
        eng.llma_rewind(0)
        assert eng.llma_generate(24, 1, 4)[0][0] == y
        got.append(y)
        assert (st.launches == 1) == (stream is None)
        eng.llma_destroy()
    assert got[0] == got[1]
