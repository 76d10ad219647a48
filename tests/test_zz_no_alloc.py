"""The allocation-free GEMM entry point gives what the allocating one gives.

Some users of this library run where they may not allocate GPU memory themselves (a host
application whose pool owns the device, a serving loop that must not stall on the allocator).
For them ``llma_gemm_rows32_bf16_noalloc`` keeps its scratch in a fixed array inside the
library.  The array is shared by all calls and remembers the previous call, so the check
is done twice in a row, with a different problem in between: stale counters or partial
tiles from one call must not leak into the next.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rand_bf16(shape, scale, seed):
    import torch
    g = torch.Generator(device="cpu").manual_seed(seed)
    return (torch.randn(shape, generator=g) * scale).to(torch.bfloat16).cuda()


def test_noalloc_matches_allocating_entry_point_twice():
    import torch
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16, llma_gemm_rows32_bf16_noalloc
    # (1000, 1024) has a ragged last tile and tiles shared by two CTAs; (512, 2816) splits each tile
    # over several CTAs, so the scratch (partials + counters) is really used
    cases = [(1000, 1024, 1), (512, 2816, 2), (1000, 1024, 3)]
    for n_out, k_in, seed in cases:
        W, a = _rand_bf16((n_out, k_in), 0.05, seed), _rand_bf16((32, k_in), 1.0, 100 + seed)
        want = torch.full((32, n_out), float("nan"), device="cuda")
        llma_gemm_rows32_bf16(W, a, want)
        for attempt in range(2):                      # two calls in a row on the same problem
            got = torch.full((32, n_out), float("nan"), device="cuda")
            llma_gemm_rows32_bf16_noalloc(W, a, got)
            assert torch.isfinite(got).all()
            # same kernel, same grid, same summation order: the tests' GEMM tolerance is 1e-4 of
            # the row scale; here the outputs are in fact identical
            scale = max(1.0, float(want.abs().max()))
            assert float((got - want).abs().max()) <= 1e-4 * scale, (n_out, k_in, attempt)
            assert torch.equal(got, want), (n_out, k_in, attempt)
    # the point of the entry point: a warmed-up call leaves the device's free memory where it was
    torch.cuda.synchronize()
    free_before, _ = torch.cuda.mem_get_info()
    llma_gemm_rows32_bf16_noalloc(W, a, got)
    torch.cuda.synchronize()
    free_after, _ = torch.cuda.mem_get_info()
    assert free_after == free_before


@pytest.mark.parametrize("sizes", [[(4096, 4096), (128, 64), (4096, 4096), (1000, 1024)]])   # grids of 148, 1, 148 and 16 CTAs in turn
def test_noalloc_scratch_serves_every_grid(sizes):
    """The hand-over slots are emptied once and then left empty by every call, whatever part of them it uses; a refused call
    in between changes nothing."""
    import torch
    from paper_2304_04487_b200 import LlmaError, llma_gemm_rows32_bf16, llma_gemm_rows32_bf16_noalloc
    for i, (n_out, k_in) in enumerate(sizes):
        W, a = _rand_bf16((n_out, k_in), 0.05, i), _rand_bf16((32, k_in), 1.0, 50 + i)
        want, got = torch.empty((32, n_out), device="cuda"), torch.full((32, n_out), float("nan"), device="cuda")
        llma_gemm_rows32_bf16(W, a, want)
        llma_gemm_rows32_bf16_noalloc(W, a, got)
        assert torch.equal(got, want), (n_out, k_in)
        flat = torch.zeros(n_out * k_in + 8, dtype=torch.bfloat16, device="cuda")
        with pytest.raises(LlmaError):
            llma_gemm_rows32_bf16_noalloc(flat[1:1 + n_out * k_in].view(n_out, k_in), a, got)


def test_noalloc_matches_oracle_directly():
    """The same entry point against the CPU oracle's matrix-vector product, with no other entry point in between."""
    import torch
    from oracle import model as OM
    from workloads import bf16_bits_from_f32, f32_from_bf16_bits
    from paper_2304_04487_b200 import llma_gemm_rows32_bf16_noalloc
    rng = np.random.default_rng(7)
    for n_out, k_in in ((200, 256), (512, 2816)):
        W = bf16_bits_from_f32((rng.standard_normal((n_out, k_in)) * 0.05).astype(np.float32))
        a = bf16_bits_from_f32(rng.standard_normal((32, k_in)).astype(np.float32))
        dev = lambda bits: torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
        out = torch.full((32, n_out), float("nan"), device="cuda")
        llma_gemm_rows32_bf16_noalloc(dev(W), dev(a), out)
        got, af = out.cpu().numpy(), f32_from_bf16_bits(a)
        for r in (0, 5, 31):
            want = OM.matvec(W, af[r])
            assert np.abs(got[r] - want).max() <= 1e-4 * max(1.0, np.abs(want).max()), (n_out, k_in, r)


def test_noalloc_rejects_sizes_beyond_its_scratch():
    import torch
    from paper_2304_04487_b200 import lib
    W, a = _rand_bf16((128, 64), 0.05, 0), _rand_bf16((32, 64), 1.0, 1)
    out = torch.zeros((32, 128), device="cuda")
    L = lib()
    # the size checks come before any pointer is used, so small buffers are safe here
    assert L.llma_gemm_rows32_bf16_noalloc(W.data_ptr(), a.data_ptr(), out.data_ptr(), 2048 * 128 + 1, 64, None) == -4
    assert L.llma_gemm_rows32_bf16_noalloc(W.data_ptr(), a.data_ptr(), out.data_ptr(), 128, 16384 + 64, None) == -4
    assert L.llma_gemm_rows32_bf16_noalloc(None, a.data_ptr(), out.data_ptr(), 128, 64, None) == -1
    assert float(out.abs().max()) == 0.0
