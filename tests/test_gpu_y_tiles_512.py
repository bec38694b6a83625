"""The y pass at 512^3 has two transform schedules (8 kz and 16 values per thread in three
stages, 16 kz and 32 values in two): the same butterflies in the same order, so the 3-D
transforms and the displacements are equal bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


def test_y_schedules_are_bit_identical():
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    n = 512
    plan = L.Plan(W.Instance(n, 1024.0, 5, W.COSMO), n_steps=64)
    x = torch.randn((n, n, n), generator=torch.Generator("cuda").manual_seed(3), device="cuda")

    def outputs():
        spec = L.lpt2_fft_r2c(plan, x)                              # Y_ONE forward
        back = L.lpt2_fft_c2r(plan, spec)                           # Y_ONE inverse
        pos = L.lpt2_displace(plan, noise=x, psi1=False, psi2=False)["pos"]   # Y_MULTI
        torch.cuda.synchronize()
        return spec, back, pos

    L.lpt2_set_tiles(plan, [8], [0])
    want = outputs()
    for ytile in (16, 0):
        L.lpt2_set_tiles(plan, [ytile], [0])
        for got, ref in zip(outputs(), want):
            assert torch.equal(got, ref), ytile
