"""Shell sums at the edges of the kernel's rounds: it holds two shells per value of a thread (8 at
16 cubed, 16 at 32 and 64 cubed, 24 at 96 cubed, 32 at 128 and 256 cubed), so counts of one round, one
more, several, one shell, and the most, with shells wider and narrower than a mode.

P(k) of seeded particles is compared with the shell means of |FFT|^2 in float64 of the density
that the same call returns, so only the transform and the sums differ.  Tolerance: the
library's 1e-4 per shell (an FP32 transform is good to ~1e-6 of the field's rms per mode, and a
shell of two modes may lie an order of magnitude or two below the rms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, n_shells", [
    (16, 1), (16, 8), (16, 9), (16, 256), (32, 7), (32, 8), (32, 16), (32, 17), (64, 16), (64, 33), (96, 24), (96, 25),
    (96, 121), (128, 16), (128, 32), (128, 33), (128, 65), (192, 23), (256, 32), (256, 33), (256, 256),
])
def test_shell_sums_at_round_edges(n, n_shells):
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W
    from oracle import lpt2

    box = 4.0 * n
    plan = L.Plan(W.Instance(n, box, 1, W.COSMO), n_steps=16)
    pos = torch.from_numpy(W.random_positions(n, box, 11)).cuda()
    r = L.lpt2_cic_pk(plan, pos=pos, density=True, n_shells=n_shells)
    dk = torch.fft.fftn(r["density"].double()).cpu().numpy()
    b = lpt2.shell_index(n, n_shells).ravel()
    sel = b >= 0
    count = np.bincount(b[sel], minlength=n_shells)
    power = np.bincount(b[sel], weights=(np.abs(dk).ravel() ** 2 * box ** 3 / float(n) ** 6)[sel], minlength=n_shells)
    assert np.array_equal(r["n_modes"].cpu().numpy(), count)
    want = np.where(count > 0, power / np.maximum(count, 1), 0.0)
    np.testing.assert_allclose(r["pk"].cpu().numpy(), want, rtol=1e-4, atol=0)
