"""A batch's launch shapes do not depend on the batches that a context ran before."""
import time

import pytest

from paper_2507_11542_gb300 import workloads as W
from helpers import AIR3D, DUBINS, lib_method, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dyn,small,large", [(AIR3D, (21, 21, 21), (101, 101, 101)), (DUBINS, (12, 12, 12, 12), (31, 31, 31, 31))])
def test_small_batch_first(dyn, small, large):
    """Eight FP32 solves in a fresh context and in one that ran a small batch of the
    same kind first: within a fifth of each other (1.4 to 2.6 times where the small
    batch's shape was kept)."""
    import torch
    from paper_2507_11542_gb300 import solver

    def batch(ctx, n, count, steps):
        spec = W.GridSpec(n, (-1.0, -1.5, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0, 2.0)[:len(n)], (2,))
        V = to_dev(W.random_field(spec, 3), "float32")
        m = lib_method(dynamics=dyn)
        ts = [steps * 0.8 / solver.step_bound(ctx, spec, m)]
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            solver.solve_batch(ctx, [spec] * count, [m] * count, [V] * count, [ts] * count)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    with solver.Context(0) as ctx:
        fresh = batch(ctx, large, 8, 20)
    with solver.Context(0) as ctx:
        batch(ctx, small, 1, 5)
        after = batch(ctx, large, 8, 20)
    assert after <= 1.2 * fresh


def test_short_batch_launches_its_own_steps():
    """Six steps of six solves: three stages and an advance a step and chain, two
    chains, and two launches a problem at the start; not a block of sixteen steps."""
    import torch
    from paper_2507_11542_gb300 import solver
    spec, V0 = W.double_integrator(61, 0.5)
    m = lib_method(dynamics=1)
    with solver.Context(0) as ctx:
        ts = [5.5 * 0.8 / solver.step_bound(ctx, spec, m)]
        V = to_dev(V0, "float32")
        for _ in range(2):
            outs, times, stats = solver.solve_batch(ctx, [spec] * 6, [m] * 6, [V] * 6, [ts] * 6)
        torch.cuda.synchronize()
    assert stats[0]["steps"] == 6
    assert stats[0]["kernel_launches"] <= 6 * 4 * 2 + 6 * 2 + 6
