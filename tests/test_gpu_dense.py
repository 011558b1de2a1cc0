"""The dense projection kernel (passes of more than 32 rows) alone, in every kind of plan it can be given, against the CPU
checker's matrix product."""
import numpy as np
import pytest

import oracle
from paper_2605_13319_b200 import synth

pytestmark = pytest.mark.gpu

# N: one row block, an odd number of them (the last odd CTA computes a copy nobody stores), a ragged last block.
# K: one stage, slices that differ by a step, a last ring stage and a last accumulator that are short, three and more
# accumulators (so that one is used again).
SIZES = [(128, 64), (384, 656), (272, 1040), (400, 2064), (640, 3200)]


@pytest.mark.parametrize("slices", [1, 2, 3, 4])
@pytest.mark.parametrize("tokens_per_cta", [16, 32, 48, 64, 80, 112, 128])
def test_dense_plans(tokens_per_cta, slices):
    import torch
    from paper_2605_13319_b200 import binding
    dev, t = torch.device("cuda", 0), tokens_per_cta
    for i, (N, K) in enumerate(SIZES):
        W = synth.normal_bf16((N, K), 17, 40 + i, 0.02)
        packed = binding.gemm_pack(torch.from_numpy(W.view(np.int16)).to(dev))
        for M in (1, 2 * t, 4 * t + 33):                    # a nearly empty block, a full one, a ragged third
            x = synth.normal_f32((M, K), 17, 80 + M, 1.0)
            want = oracle.linear(W, x.astype(np.float64))
            # tokens beyond M are never written: whatever they hold must not matter
            scratch = torch.full((binding.lib().pipesd_debug_gemm_dense_scratch_bytes(M, K, t),), 255, dtype=torch.uint8, device=dev)
            y = torch.full((M, N), float("nan"), device=dev)
            for _ in range(3):
                binding.debug_gemm_dense(packed, torch.from_numpy(x).to(dev), y, scratch, N, K, t, slices)
            torch.cuda.synchronize()
            # fp32 accumulation of K products of |w| ~ 0.02, |x| ~ 1, activations carried as bf16 hi + lo (2^-17): as in the
            # small-M kernel's test
            assert np.abs(y.cpu().numpy() - want).max() < 3e-5 * 0.02 * np.sqrt(K) * 4, (N, K, M)


@pytest.mark.parametrize("N,K", [(256, 256), (272, 688), (512, 1024), (2048, 2048), (4096, 4096)])
def test_dense_sums_as_exact_as_small_m(N, K):
    """The tensor pipe truncates where it adds, so depth costs precision: the rms error of rows through this kernel may not
    exceed the small-M kernel's, whose K slices are an eighth of K here (5 % for another order of sums)."""
    import torch
    from paper_2605_13319_b200 import binding
    dev, M = torch.device("cuda", 0), 32
    W = synth.normal_bf16((N, K), 19, 5, 0.02)
    packed = binding.gemm_pack(torch.from_numpy(W.view(np.int16)).to(dev))
    x = synth.normal_f32((M, K), 19, 6, 1.0)
    want = oracle.linear(W, x.astype(np.float64))
    xd, y = torch.from_numpy(x).to(dev), torch.empty((M, N), device=dev)

    def rms():
        torch.cuda.synchronize()
        return np.sqrt(np.mean((y.cpu().numpy() - want) ** 2))

    binding.gemm_run(packed, xd, y, binding.gemm_scratch(M, N, K, dev), N, K)
    small = rms()
    scratch = torch.zeros(binding.lib().pipesd_debug_gemm_dense_scratch_bytes(M, K, 16), dtype=torch.uint8, device=dev)
    binding.debug_gemm_dense(packed, xd, y, scratch, N, K, 16, 1)
    dense = rms()
    print(f"rms error {N} x {K}: small-M {small:.3e}, dense {dense:.3e}")
    assert dense < 1.05 * small


def test_dense_rejects_bad_plans():
    from paper_2605_13319_b200 import binding
    L = binding.lib()
    for M, N, K, t, s in [(0, 128, 128, 16, 1), (8, 120, 128, 16, 1), (8, 128, 100, 16, 1), (8, 128, 128, 8, 1), (8, 128, 128, 24, 1),
                          (8, 128, 128, 144, 1), (8, 128, 128, 16, 0), (8, 128, 128, 16, 5), (8, 128, 32, 16, 3)]:
        assert L.pipesd_debug_gemm_dense(1, 1, 1, 1, M, N, K, t, s, None) == binding.E_INVALID
    assert L.pipesd_debug_gemm_dense_scratch_bytes(33, 64, 16) == 2 * 32 * 64 * 4
    assert L.pipesd_debug_gemm_dense_scratch_bytes(33, 64, 24) == 0
