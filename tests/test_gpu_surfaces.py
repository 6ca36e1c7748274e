"""Initial surfaces on grids of every form: one node a thread on small, thin and
(FP64) one-dimensional grids, rows of four nodes a thread on the others, lists of
primitives longer than the unrolled four, primitives that span some of the
dimensions. Against the oracle, with the bounds of test_gpu_implicit.py (unit
roundoff times the terms of a sum, whatever the number of primitives: they are
joined by exact minima and maxima)."""
import numpy as np
import pytest

from oracle import implicit as I
from paper_2507_11542_gb300 import workloads as W
from helpers import to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11542_gb300 import solver
    with solver.Context(0) as c:
        yield c


def _shapes(ndim, count):
    r = np.random.default_rng(count)
    out = []
    for k in range(count):
        dims = tuple(d for d in range(ndim) if r.uniform() < 0.7) or (int(r.integers(ndim)),)
        out.append({"kind": (I.SPHERE, I.RECTANGLE, I.ELLIPSOID)[int(r.integers(3))],
                    "op": (I.UNION, I.INTERSECT, I.SUBTRACT)[int(r.integers(3))], "dims": dims,
                    "center": tuple(r.uniform(-0.8, 0.8, ndim)), "axes": tuple(r.uniform(0.2, 2.0, ndim)),
                    "radius": float(r.uniform(0.2, 1.2))})
    return out


@pytest.mark.parametrize("n", [(127,), (129,), (65537,), (70000,), (300000,), (1, 9), (5, 3), (257, 255), (257, 256),
                               (512, 512), (1025, 257), (3, 90001), (90001, 3), (4, 4, 5000), (31, 3, 801), (64, 64, 65),
                               (33, 2, 2001), (4, 5, 6, 7), (17, 16, 16, 16), (3, 3, 100, 81), (23, 22, 23, 24)])
@pytest.mark.parametrize("count", [1, 5, 32])
@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_surface_of_any_grid_and_list(ctx, n, count, dtype):
    from paper_2507_11542_gb300 import solver
    D = len(n)
    g = W.GridSpec(n, (-1.2, -1.0, -0.8, -1.1)[:D], (1.1, 1.3, 0.9, 1.0)[:D], (0,) if n[0] == 1 else ())
    shapes = _shapes(D, count)
    got = to_host(solver.implicit_surface(ctx, g, shapes, dtype), g.n)
    ref = I.implicit_surface(g, shapes)
    tol = 1e-14 if dtype == "float64" else 1e-6
    assert np.max(np.abs(got - ref)) <= tol * float(np.max(np.abs(ref)))


@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_one_dimension_costs_what_two_do(ctx, dtype):
    """4 M nodes of one line, and of 2000 lines: at most twice the time (a block
    whose threads have one row to share took nine times in FP64)."""
    import torch
    from paper_2507_11542_gb300 import solver
    took = []
    for n in ((4000000,), (2000, 2000)):
        g = W.GridSpec(n, (-1.0,) * len(n), (1.0,) * len(n))
        shapes = [{"kind": I.SPHERE, "dims": (0,), "center": (0.1,) * len(n), "radius": 0.4}] * 4
        out = torch.empty(4000000, dtype=getattr(torch, dtype), device="cuda")
        best = 1e9
        for rep in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                solver.implicit_surface(ctx, g, shapes, out.dtype, out=out)
            b.record()
            torch.cuda.synchronize()
            if rep:
                best = min(best, a.elapsed_time(b))
        took.append(best)
    assert took[0] <= 2.0 * took[1]
