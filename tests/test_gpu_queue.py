"""Stage kernels that start before the kernel in front of them has ended: a long
row of steps in a stream runs as fast per step as a short one."""
import pytest

from paper_2507_11542_gb300 import workloads as W
from helpers import AIR3D, DI, PARAMS, lib_method, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dyn,n,periodic,scheme", [(DI, (40, 1000), (), 3), (DI, (101, 101), (), 5),
                                                    (AIR3D, (21, 21, 21), (2,), 3), (AIR3D, (41, 41, 41), (2,), 5)])
def test_steps_in_flight_do_not_slow_each_other(dyn, n, periodic, scheme):
    """128 steps at once and 4 at once, FP64, from a GPU that is kept busy while
    they are enqueued; kernels that wait on an SM for several others in front of
    them cost twice the time (30 and 65 us a step of 40 x 1000). A fifth more is
    well above what two runs differ by."""
    import torch
    from paper_2507_11542_gb300 import solver
    spec = W.GridSpec(n, (-1.0, -1.5, 0.0)[:len(n)], (2.0, 1.0, 6.0)[:len(n)], periodic)
    V = to_dev(W.random_field(spec, 4))
    m = lib_method(scheme=scheme, dynamics=dyn)
    with solver.Context(0) as ctx:
        for _ in range(20):
            solver.rk3_step(ctx, spec, m, V, 1e-6)

        def per_step(count):
            best = 1e9
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                torch.cuda._sleep(4000000)
                a.record()
                for _ in range(count):
                    solver.rk3_step(ctx, spec, m, V, 1e-6)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) / count)
            return best

        assert per_step(128) <= 1.2 * per_step(4)
