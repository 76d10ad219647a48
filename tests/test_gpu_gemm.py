"""The projection kernel on its own, against the CPU oracle's matrix-vector product."""
import numpy as np
import pytest

from oracle import model as OM
from workloads import bf16_bits_from_f32, f32_from_bf16_bits

pytestmark = pytest.mark.gpu


def _case(n_out, k_in, seed):
    rng = np.random.default_rng(seed)
    W = bf16_bits_from_f32((rng.standard_normal((n_out, k_in)) * 0.05).astype(np.float32))
    a = bf16_bits_from_f32(rng.standard_normal((32, k_in)).astype(np.float32))
    return W, a


def _to_dev(bits):
    import torch
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


# shapes: one tile; several tiles with a ragged last one; k split over several CTAs; wide k
@pytest.mark.parametrize("n_out,k_in", [(128, 64), (200, 256), (1000, 1024), (512, 2816), (4096, 4096)])
def test_gemm_rows32_matches_oracle(n_out, k_in):
    import torch
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16
    W, a = _case(n_out, k_in, seed=n_out + k_in)
    out = torch.full((32, n_out), float("nan"), device="cuda", dtype=torch.float32)
    llma_gemm_rows32_bf16(_to_dev(W), _to_dev(a), out)
    got = out.cpu().numpy()
    af = f32_from_bf16_bits(a)
    rows = range(32) if n_out * k_in <= 1 << 21 else (0, 7, 31)       # sampled rows at the large sizes
    for r in rows:
        want = OM.matvec(W, af[r])
        # fp32 accumulation of k_in products of magnitude ~0.05: error far below 1e-4 of the row's scale
        assert np.abs(got[r] - want).max() <= 1e-4 * max(1.0, np.abs(want).max()), (r, np.abs(got[r] - want).max())
    assert np.isfinite(got).all()
    # same bits on a second run (fixed summation order over the CTAs that share a tile)
    out2 = torch.empty_like(out)
    llma_gemm_rows32_bf16(_to_dev(W), _to_dev(a), out2)
    assert torch.equal(out, out2)


def test_gemm_rejects_bad_arguments():
    import torch
    from paper_2304_04487_b200 import LlmaError, lib
    W, a = _case(128, 64, 0)
    Wd, ad = _to_dev(W), _to_dev(a)
    out = torch.empty((32, 128), device="cuda")
    L = lib()
    assert L.llma_gemm_rows32_bf16(None, ad.data_ptr(), out.data_ptr(), 128, 64, None) == -1
    assert L.llma_gemm_rows32_bf16(Wd.data_ptr(), ad.data_ptr(), out.data_ptr(), 128, 96, None) == -9
    assert L.llma_gemm_rows32_bf16(Wd.data_ptr(), ad.data_ptr(), out.data_ptr(), 0, 64, None) == -9


@pytest.mark.parametrize("threads", [2, 6, 20])            # fewer and more than the scratch blocks kept between calls
def test_gemm_concurrent_calls(threads):
    """Calls from several threads on streams of their own: each has scratch of its own, and it stays usable."""
    import threading
    import torch
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16
    work, want = [], []
    for i in range(threads):
        W, a = _case(512 + 128 * i, 2816, seed=50 + i)     # every tile is shared by several CTAs
        Wd, ad = _to_dev(W), _to_dev(a)
        out = torch.empty((32, W.shape[0]), device="cuda")
        llma_gemm_rows32_bf16(Wd, ad, out)
        work.append((Wd, ad)); want.append(out.clone())
    torch.cuda.synchronize()
    bad = []

    def call(i):
        st, out = torch.cuda.Stream(), torch.empty_like(want[i])
        for _ in range(20):
            llma_gemm_rows32_bf16(*work[i], out, stream=st)
            if not torch.equal(out, want[i]):
                bad.append(i)
    ts = [threading.Thread(target=call, args=(i,)) for i in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad


@pytest.mark.parametrize("n_out,k_in", [(128, 64), (200, 192), (1000, 1024)])
@pytest.mark.parametrize("shift", [1, 2, 4, 7])
def test_rows_off_the_16_byte_grid(n_out, k_in, shift):
    """The activation rows may lie anywhere (2-byte aligned), the result on any fp32: same bits as on a boundary."""
    import torch
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16, llma_gemm_rows32_bf16_noalloc
    W, a = (_to_dev(x) for x in _case(n_out, k_in, seed=9))
    want = torch.empty((32, n_out), device="cuda")
    llma_gemm_rows32_bf16(W, a, want)
    flat = torch.empty(32 * k_in + shift, device="cuda", dtype=torch.bfloat16)
    flat[shift:] = a.flatten()
    rows = flat[shift:].view(32, k_in)
    assert rows.data_ptr() % 16
    for gemm in (llma_gemm_rows32_bf16, llma_gemm_rows32_bf16_noalloc):
        res = torch.zeros(32 * n_out + 1, device="cuda")
        gemm(W, rows, res[1:].view(32, n_out))
        assert torch.equal(res[1:].view(32, n_out), want)


def test_misaligned_operands_are_rejected():
    import torch
    from paper_2304_04487_b200 import lib
    W, a = (_to_dev(x) for x in _case(128, 64, 0))
    out = torch.empty(32 * 128 + 1, device="cuda")
    for gemm in (lib().llma_gemm_rows32_bf16, lib().llma_gemm_rows32_bf16_noalloc):
        assert gemm(W.data_ptr() + 2, a.data_ptr(), out.data_ptr(), 64, 64, None) == -9
        assert gemm(W.data_ptr(), a.data_ptr() + 1, out.data_ptr(), 128, 64, None) == -9
        assert gemm(W.data_ptr(), a.data_ptr(), out.data_ptr() + 2, 128, 64, None) == -9


def test_scratch_outlives_all_but_the_last_engine():
    """The product's scratch between calls: other engines' coming and going leaves it alone, the last one takes it along."""
    import os
    import subprocess
    import sys
    code = """
import torch
from paper_2304_04487_b200 import Engine, llma_gemm_rows32_bf16
from workloads import SHAPES, make_weights
shape = SHAPES["tiny-fp32"]
w = make_weights(shape, seed=0)
free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]
W, a, out = torch.ones(512, 2816, device="cuda").bfloat16(), torch.ones(32, 2816, device="cuda").bfloat16(), torch.empty(32, 512, device="cuda")
A = Engine(shape, w, max_seq=64, max_ref=8, max_k=1)
B = Engine(shape, w, max_seq=64, max_ref=8, max_k=1)
llma_gemm_rows32_bf16(W, a, out)
A.llma_destroy()
before = free()
llma_gemm_rows32_bf16(W, a, out)
assert free() == before, "scratch was allocated anew although an engine is left"
C = Engine(shape, w, max_seq=64, max_ref=8, max_k=1)
C.llma_destroy()
B.llma_destroy()
idle = free()
llma_gemm_rows32_bf16(W, a, out)
assert free() < idle, "scratch was kept past the last engine"
assert float(out[0, 0]) == 2816.0
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)
