"""CIC weights of particles that leave their block of 16 Lagrangian cells by more than four cells
(upwards along z: seven) are summed in FP32 (the nearer ones in units of 2^-19).  The last layer of
every block along one axis is moved beyond that by a fraction of a cell, every other particle stays on its lattice point (weight 1, exact
in either form), so the cells that the layer reaches hold one exact weight and four FP32 ones:
against float64, five additions within 2^-24 of the sum, two products within 2^-24 of each weight
and the contrast's subtraction within 2^-24 are 2^-21 of the density at most."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis, shift, layer", [(0, 5, 15), (0, -5, 0), (1, 5, 15), (1, -5, 0), (2, 8, 15), (2, -5, 0)])
def test_far_weights_are_fp32(axis, shift, layer):
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    n = 64   # cells of 1: positions are in cells, multiples of 2^-18, exact
    gen = torch.Generator("cuda").manual_seed(axis + 7)
    grid = torch.arange(n, device="cuda", dtype=torch.float64)
    pos = torch.stack(torch.meshgrid(grid, grid, grid, indexing="ij"))
    frac = torch.randint(1, 2 ** 18, (3, n, n, n), generator=gen, device="cuda").double() * 2.0 ** -18
    frac[axis] += shift
    pos = torch.where(pos[axis] % 16 == layer, (pos + frac) % n, pos)
    plan = L.Plan(W.Instance(n, float(n), 1, W.COSMO), n_steps=16)
    got = L.lpt2_cic_pk(plan, pos=pos.float(), density=True, n_shells=8)["density"].double() + 1.0
    assert torch.equal(pos.float().double(), pos)
    cell = pos.floor().long()
    d = pos - cell
    want = torch.zeros(n * n * n, device="cuda", dtype=torch.float64)
    for cx in (0, 1):
        for cy in (0, 1):
            for cz in (0, 1):
                w = 1.0
                for a, c in enumerate((cx, cy, cz)):
                    w = w * (d[a] if c else 1.0 - d[a])
                i = (((cell[0] + cx) % n) * n + (cell[1] + cy) % n) * n + (cell[2] + cz) % n
                want.index_add_(0, i.reshape(-1), w.reshape(-1))
    want = want.view(n, n, n)
    assert float(((got - want).abs() - 2.0 ** -21 * want).max()) <= 0.0
