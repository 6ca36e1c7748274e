"""The launch shape that hj_rk3_step_static takes without timing, beside the one
that hj_rk3_step has timed."""
import pytest

from paper_2507_11542_gb300 import workloads as W
from helpers import AIR3D, DUBINS, NORM, lib_method, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dyn,n,periodic,dtype,scheme", [
    (NORM, (101, 101, 101), (), "float64", 3), (AIR3D, (101, 101, 101), (2,), "float64", 5), (AIR3D, (41, 41, 41), (2,), "float64", 1),
    (DUBINS, (15, 15, 15, 15), (2,), "float64", 3), (DUBINS, (31, 31, 31, 31), (2,), "float32", 5), (AIR3D, (61, 61, 61), (2,), "float32", 2)])
def test_shape_taken_without_timing(ctx, dyn, n, periodic, dtype, scheme):
    """At most 1.35 times the timed shape's step (a fixed shape took 1.5 to 1.9
    times on these grids; the model's first is 4 to 6 % above the best on average
    and 16 % at most over the grids it was held against), and the same bits."""
    import torch
    from paper_2507_11542_gb300 import _lib as L, solver
    spec = W.GridSpec(n, (-1.0, -1.5, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0, 2.0)[:len(n)], periodic)
    m = lib_method(scheme=scheme, dynamics=dyn)
    grid = L.make_grid(spec)
    V = to_dev(W.random_field(spec, 4), dtype)
    stream = torch.cuda.current_stream().cuda_stream
    steps = [lambda t: solver.rk3_step(ctx, spec, m, t, 1e-6),
             lambda t: L.hj_rk3_step_static(stream, 0, grid, m, L.dtype_code(t.dtype), t, 1e-6)]
    out, took = [], []
    for step in steps:
        t = V.clone()
        step(t)
        out.append(t)
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            torch.cuda._sleep(1000000)
            a.record()
            for _ in range(20):
                step(t)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        took.append(best)
    assert torch.equal(out[0], out[1])
    assert took[1] <= 1.35 * took[0]


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11542_gb300 import solver
    with solver.Context(0) as c:
        yield c
