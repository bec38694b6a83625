"""Pencils of 32, 128 and 512 points have two stage sequences (three stages, whose middle radix may
run on warp shuffles, or two), chosen per pass.  The 3-D transforms use both: the z passes one, the
y and x passes the other.  Against torch's float64 transform, relative L2 error: an FP32 transform
rounds once or twice per radix-2 level of its log2(n^3), so 2 x 2^-24 x log2(n^3) bounds it."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 128, 512])
def test_both_stage_sequences(n):
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    plan = L.Plan(W.Instance(n, 2.0 * n, 1, W.COSMO), n_steps=16)
    x = torch.randn((n, n, n), generator=torch.Generator("cuda").manual_seed(n), device="cuda")
    tol = 2.0 * 2.0 ** -24 * math.log2(float(n) ** 3)
    got = L.lpt2_fft_r2c(plan, x)
    want = torch.fft.rfftn(x.double())[..., : n // 2]
    assert float(torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want)) < tol
    # back (unnormalised), the kz = n/2 plane zero
    full = torch.zeros((n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
    full[..., : n // 2] = got
    want = torch.fft.irfftn(full, s=(n, n, n), norm="forward")
    back = L.lpt2_fft_c2r(plan, got).double()
    assert float(torch.linalg.vector_norm(back - want) / torch.linalg.vector_norm(want)) < tol


@pytest.mark.parametrize("count", [1, 2, 3, 255, 2 * 152 * 4 * 256 + 1])
def test_box_muller_counts(count):
    """Two draws per thread: an odd count leaves the last thread one; the draws are those of a longer call."""
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    plan = L.Plan(W.Instance(16, 64.0, 1, W.COSMO), n_steps=16)
    g = torch.Generator("cuda").manual_seed(9)
    words = torch.randint(-2 ** 31, 2 ** 31, (count + 5, 2), generator=g, device="cuda").to(torch.int32)
    assert torch.equal(L.lpt2_box_muller(plan, words[:count].contiguous()), L.lpt2_box_muller(plan, words)[:count])
