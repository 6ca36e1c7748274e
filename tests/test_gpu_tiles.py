"""Tiles of the row kernel at the sizes where they can go wrong: segments along
dimension 0 (at most 124 nodes), one and two rows in the last tile, rows shorter
than a warp, the least and an odd number of planes, ghost rows and columns that
begin inside a halo. Held against the oracle (FP64) and against the
one-node-per-thread kernel, which has no tiles (FP32)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_11542_gb300 import workloads as W
from helpers import lib_method, oracle_method, rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu

DI, AIR3D, DUBINS, NORM = 1, 2, 3, 4


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11542_gb300 import solver
    with solver.Context(0) as c:
        yield c


def _grid(n, periodic):
    lo = (-1.0, -1.5, 0.0, 0.0)[:len(n)]
    hi = (2.0, 1.0, 6.0, 2.0)[:len(n)]
    return W.GridSpec(tuple(n), lo, hi, periodic)


@pytest.mark.parametrize("dyn,n,periodic", [
    (DI, (124, 9), ()), (DI, (125, 10), (0,)), (DI, (249, 4), (1,)), (DI, (4, 17), ()), (DI, (33, 11), (0, 1)),
    (NORM, (125, 8, 4), ()), (NORM, (5, 10, 7), (0, 1, 2)), (NORM, (31, 9, 5), (1,)), (AIR3D, (126, 5, 6), (2,)),
    (AIR3D, (61, 25, 4), (2,)), (DUBINS, (37, 9, 5, 4), (2,)), (DUBINS, (4, 10, 4, 5), (0, 1, 2, 3)),
])
@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("scheme", [5, 2])
def test_tile_edges(ctx, dyn, n, periodic, dtype, scheme):
    from paper_2507_11542_gb300 import solver
    spec = _grid(n, periodic)
    V = W.random_field(spec, 5)
    dt = 0.5 / O.step_bound_inv(spec, oracle_method(dynamics=dyn))
    got = to_dev(V, dtype)
    solver.rk3_step(ctx, spec, lib_method(scheme=scheme, dynamics=dyn, brt=1, kernel=1), got, dt)
    if dtype == "float64":
        want = O.rk3_step(spec, oracle_method(scheme=scheme, dynamics=dyn, brt=1), V, dt)
        assert rel_err(to_host(got, spec.n), want) <= 1e-12
    else:
        node = to_dev(V, dtype)
        solver.rk3_step(ctx, spec, lib_method(scheme=scheme, dynamics=dyn, brt=1, kernel=2), node, dt)
        assert rel_err(to_host(got, spec.n), to_host(node, spec.n)) <= 1e-5
    for ty in (1, 2, 3):  # pinned rows give the same bits
        if (n[0] + 1) * ty > (512 if dtype == "float64" else 1024) or ty > min(n[0], n[1]):
            continue
        again = to_dev(V, dtype)
        solver.rk3_step(ctx, spec, lib_method(scheme=scheme, dynamics=dyn, brt=1, kernel=1, tile=[ty, 2, 1, 0]), again, dt)
        np.testing.assert_array_equal(to_host(again, spec.n), to_host(got, spec.n))
