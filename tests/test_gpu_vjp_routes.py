"""The adjoint skips the passes of cotangents that are not given; the route with every pass is
taken when they are given as zeros.  Both must agree: the same numbers are transformed, with
zeros added, so bit for bit in the noise gradient except where a zero is added to a rounded
number (none is: the density cotangent and the gathered gradient are exactly zero or exactly
g_density).  P(k) cotangents of zero leave g_density plus a transform of zeros."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, keep", [(16, False), (32, True), (96, False), (128, False)])
def test_absent_cotangents_equal_zero_cotangents(n, keep):
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    ns = 12
    plan = L.Plan(W.Instance(n, 3.0 * n, 1, W.COSMO), n_steps=64, keep_state=keep)
    gen = torch.Generator("cuda").manual_seed(n)
    noise = torch.randn((n, n, n), generator=gen, device="cuda")
    g_pos = torch.randn((3, n, n, n), generator=gen, device="cuda")
    g_den = torch.randn((n, n, n), generator=gen, device="cuda")
    zero_pk = torch.zeros(ns, dtype=torch.float64, device="cuda")
    shifted = torch.empty(n ** 3 + 1, device="cuda")[1:].view(n, n, n)   # 4-byte aligned copy
    shifted.copy_(g_den)

    def grad(**kw):
        if keep:
            L.lpt2_displace(plan, noise=noise, psi1=False, psi2=False, pos=False)
        g, t = L.lpt2_displace_vjp(plan, noise=noise, n_shells=ns, **kw)
        torch.cuda.synchronize()
        return g, t

    full = grad(g_pos=g_pos, g_density=torch.zeros_like(g_den), g_pk=zero_pk)
    assert all(torch.equal(a, b) for a, b in zip(grad(g_pos=g_pos), full))
    full = grad(g_density=g_den, g_pk=zero_pk)
    assert all(torch.equal(a, b) for a, b in zip(grad(g_density=g_den), full))
    assert all(torch.equal(a, b) for a, b in zip(grad(g_density=shifted), full))
    nothing = grad()
    assert float(nothing[0].abs().max()) == 0.0 and float(nothing[1]) == 0.0


def test_position_cotangent_keeps_the_density():
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    n = 32
    plan = L.Plan(W.Instance(n, 96.0, 1, W.COSMO), n_steps=64)
    noise = torch.randn((n, n, n), generator=torch.Generator("cuda").manual_seed(4), device="cuda")
    g_pos = torch.ones((3, n, n, n), device="cuda")
    L.lpt2_displace(plan, noise=noise, psi1=False, psi2=False, pos=False)
    want = L.lpt2_cic_pk(plan, density=True, n_shells=8)
    L.lpt2_displace_vjp(plan, noise=noise * 2, g_pos=g_pos)
    got = L.lpt2_cic_pk(plan, density=True, n_shells=8)
    assert torch.equal(got["density"], want["density"]) and torch.equal(got["pk"], want["pk"])
