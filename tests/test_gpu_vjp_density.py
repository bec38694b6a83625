"""The density that lpt2_cic_pk(plan, NULL, ...) reads after an adjoint with a cotangent of the
positions alone: that of the last lpt2_displace while the workspace holds it, otherwise the one of
the adjoint's own forward map, as with any other cotangent.  The workspace starts as NaN, so a
density that nobody deposited shows.  It is compared with that of lpt2_displace on the same noise:
the same kernels, whose float reductions may add in another order, at most 32 to a cell, each
rounded by 2^-20 at contrasts below 31, on either side: 2^-14.  P(k) to the library's 1e-4."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

NS = 8


def _blank(plan):
    from paper_1909_06282_gb300 import _lib

    plan.workspace.fill_(0xff)   # NaN in every float
    assert _lib.load_library().lpt2_set_workspace(plan.handle, C.c_void_p(plan.workspace.data_ptr()),
                                                  plan.workspace.numel()) == 0


def _case(n=32, **kw):
    import torch

    import paper_1909_06282_gb300 as L
    import workloads as W

    plan = L.Plan(W.Instance(n, 4.0 * n, 1, W.COSMO), n_steps=32, **kw)
    _blank(plan)
    gen = torch.Generator("cuda").manual_seed(n)
    noise = [torch.randn((n, n, n), generator=gen, device="cuda") for _ in range(3)]
    g_pos = torch.randn((3, n, n, n), generator=gen, device="cuda")
    pos = torch.from_numpy(W.random_positions(n, 4.0 * n, 3)).cuda()
    return L, plan, noise, g_pos, pos


def _density(L, plan):
    r = L.lpt2_cic_pk(plan, density=True, n_shells=NS)
    return r["density"], r["pk"]


def _of(L, plan, noise):
    L.lpt2_displace(plan, noise=noise, psi1=False, psi2=False, pos=False)
    return _density(L, plan)


def _same(a, b):
    import torch

    assert float(b[0].max()) < 31.0
    torch.testing.assert_close(a[0], b[0], rtol=0.0, atol=2.0 ** -14)
    torch.testing.assert_close(a[1], b[1], rtol=1e-4, atol=0.0)


@pytest.mark.parametrize("keep", [False, True])
def test_adjoint_without_a_displaced_density_deposits_its_own(keep):
    L, plan, noise, g_pos, _ = _case(keep_state=keep)
    got = []
    for q in noise[:2]:   # the second call finds the first one's density, which is not its own
        L.lpt2_displace_vjp(plan, noise=q, g_pos=g_pos, n_shells=NS)
        got.append(_density(L, plan))
    for q, r in zip(noise, got):
        _same(r, _of(L, plan, q))


@pytest.mark.parametrize("between", ["cic_pk", "cic_pk_est", "vjp", "autotune", "workspace"])
def test_a_replaced_density_is_not_taken_for_the_displaced_one(between):
    L, plan, noise, g_pos, pos = _case()
    a = _of(L, plan, noise[0])
    L.lpt2_displace_vjp(plan, noise=noise[1], g_pos=g_pos, n_shells=NS)
    _same(_density(L, plan), a)
    if between == "cic_pk":
        L.lpt2_cic_pk(plan, pos=pos, n_shells=NS)
    elif between == "cic_pk_est":
        L.lpt2_cic_pk_est(plan, pos=pos, n_shells=NS)
    elif between == "vjp":
        L.lpt2_displace_vjp(plan, noise=noise[2], g_density=g_pos[0].contiguous(), n_shells=NS)
    elif between == "autotune":
        L.lpt2_autotune(plan, n_shells=NS, reps=1)
    else:
        _blank(plan)
    L.lpt2_displace_vjp(plan, noise=noise[1], g_pos=g_pos, n_shells=NS)
    _same(_density(L, plan), _of(L, plan, noise[1]))


def test_captured_adjoint_deposits():
    import torch

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        L, plan, noise, g_pos, pos = _case()
        L.lpt2_displace_vjp(plan, noise=noise[1], g_pos=g_pos, n_shells=NS)
        _of(L, plan, noise[0])
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            L.lpt2_displace_vjp(plan, noise=noise[1], g_pos=g_pos, n_shells=NS)
        L.lpt2_cic_pk(plan, pos=pos, n_shells=NS)
        graph.replay()
        _same(_density(L, plan), _of(L, plan, noise[1]))
        s.synchronize()


@pytest.mark.parametrize("cotangent", ["g_pos", "g_density"])
def test_every_adjoint_makes_the_shell_geometry(cotangent):
    """So that a P(k) call captured after it holds the estimator's kernels only."""
    L, plan, noise, g_pos, _ = _case()
    g = g_pos if cotangent == "g_pos" else g_pos[0].contiguous()
    L.lpt2_displace_vjp(plan, noise=noise[0], n_shells=NS, **{cotangent: g})
    count = [L.lpt2_launch_count(plan)]
    for _ in range(2):
        _density(L, plan)
        count.append(L.lpt2_launch_count(plan))
    assert count[1] - count[0] == count[2] - count[1]
