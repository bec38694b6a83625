"""The growth kernel at the edges of its chunks and blocks: step counts around a multiple of
the chunk (8 steps), one step, table lengths around a multiple of the four k of a block, the
smallest tables, every source geometry, and GR.

Tolerance: the kernel takes the oracle's RK4 steps (same step count) in FP64 with another
order of operations.  Each step rounds a state a few dozen times at 1.1e-16; 1024 steps that
all round one way give 1024 * 40 * 1.1e-16 = 4.5e-12 of the largest value, the bar is 1e-11."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_steps, n_k, variant, fr0, a_out", [
    (1, 2, 0, 1e-5, 1.0), (7, 3, 0, 1e-5, 1.0), (8, 4, 0, 1e-4, 0.5), (9, 5, 0, 1e-6, 1.0),
    (15, 7, 1, 1e-5, 1.0), (17, 9, 4, 1e-5, 0.35), (33, 6, 8, 1e-5, 1.0), (250, 130, 5, 1e-6, 1.0),
    (250, 513, 6, 1e-5, 1.0), (250, 31, 9, 1e-5, 0.7), (1023, 65, 0, 0.0, 1.0), (1024, 512, 3, 1e-4, 1.0),
])
def test_tables_at_chunk_and_block_edges(n_steps, n_k, variant, fr0, a_out):
    import paper_1909_06282_gb300 as L
    import workloads as W
    from oracle import growth

    c = W.COSMO.replace(fr0_abs=fr0, d2_variant=variant)
    plan = L.Plan(W.Instance(16, 64.0, 1, c, a_out=a_out), n_steps=n_steps, n_k=n_k, workspace=False)
    got = [t.cpu().numpy() for t in L.lpt2_growth_tables(plan)]
    ref = growth.growth_tables(c, a_out, k=growth.k_table(n_k), n_steps=n_steps)
    for g, key in zip(got, ("D1", "D2", "dD1", "dD2")):
        scale = np.max(np.abs(ref[key]))
        assert np.max(np.abs(g - ref[key])) <= 1e-11 * max(scale, 1e-300), key
