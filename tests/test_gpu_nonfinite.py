"""Infinite values in a field that is stepped (an obstacle, or a node that is
never reached, marked +inf or -inf), and values near the largest: the
combination cv V^n + cu w of stages 2 and 3 keeps an infinite value infinite and
a representable one finite. hj_solve refuses such fields; the single step and
stage take them.

The field is constant but for the marked nodes and the rule is min(0, .), so
that the term is 0 at every node (WENO5 of a constant, or NaN, which min(0, .)
takes for 0) and w = u: the expected result is known exactly, up to the
combination's own rounding (three of them, 2^-24 of the largest term each)."""
import numpy as np
import pytest

from paper_2507_11542_gb300 import workloads as W
from helpers import AIR3D, DI, DUBINS, NORM, lib_method, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11542_gb300 import solver
    with solver.Context(0) as c:
        yield c


GRIDS = {DI: ((37, 29), ()), NORM: ((21, 18), (1,)), AIR3D: ((35, 19, 16), (2,)), DUBINS: ((13, 11, 9, 7), (2,))}


@pytest.mark.parametrize("dyn", [DI, NORM, AIR3D, DUBINS])
@pytest.mark.parametrize("kernel,tile", [(0, (0, 0, 0, 0)), (1, (3, 2, 0, 0)), (2, (0, 0, 0, 0))])
@pytest.mark.parametrize("mark", [np.inf, -np.inf, 3e38, -3e38])
@pytest.mark.parametrize("stage", [2, 3])
def test_stage_keeps_infinite_and_largest_values(ctx, dyn, kernel, tile, mark, stage):
    import torch
    from paper_2507_11542_gb300 import solver
    n, periodic = GRIDS[dyn]
    spec = W.GridSpec(n, (-1.0, -1.5, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0, 2.0)[:len(n)], periodic)
    rng = np.random.default_rng(3)
    u = np.full(n, 1.25)
    u[rng.uniform(size=n) < 0.02] = mark
    old = np.float32(rng.uniform(-2.0, 2.0, size=n)).astype(np.float64)
    old[rng.uniform(size=n) < 0.02] = mark
    old[rng.uniform(size=n) < 0.02] = -mark if np.isfinite(mark) else mark
    ud, vn = to_dev(u, "float32"), to_dev(old, "float32")
    out = torch.empty_like(ud)
    solver.rk3_stage(ctx, spec, lib_method(dynamics=dyn, brt=1, kernel=kernel, tile=tile), stage, ud, vn, out, 0.004)
    cv, cu = ((0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))[stage - 2]
    u, old = np.float32(u).astype(np.float64), np.float32(old).astype(np.float64)
    want = cv * old + cu * u
    got = to_host(out, n)
    inf = np.isinf(want)
    np.testing.assert_array_equal(got[inf], want[inf])
    err = np.abs(got[~inf] - want[~inf])
    assert (err <= 3 * 2.0 ** -24 * (np.abs(old[~inf]) + np.abs(u[~inf]))).all()


@pytest.mark.parametrize("dyn", [DI, NORM, AIR3D, DUBINS])
@pytest.mark.parametrize("mark", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("scheme", [1, 2, 3, 5])
@pytest.mark.parametrize("tile", [(0, 0, 0, 0), (3, 2, 0, 0)])
def test_fp64_rule_leaves_nan(ctx, dyn, mark, scheme, tile):
    """min(0, .) of a term that is NaN is NaN in FP64, as in the oracle: nodes beside
    infinite or undefined ones do not look like nodes where nothing moves. Held on
    the same nodes as the oracle's, but WENO5 of infinite data, whose weights the two
    form differently (infinite or NaN), and ENO2/3 of NaN data, whose candidates the
    kernel compares by their bits (NaN above everything, so that the other one is
    taken; the oracle's comparison with NaN takes the right one)."""
    from oracle import oracle as O
    from paper_2507_11542_gb300 import solver
    from helpers import oracle_method
    n, periodic = GRIDS[dyn]
    spec = W.GridSpec(n, (-1.0, -1.5, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0, 2.0)[:len(n)], periodic)
    V = np.asfortranarray(W.random_field(spec, 6))
    V[np.random.default_rng(4).uniform(size=n) < 0.01] = mark
    with np.errstate(all="ignore"):
        want = O.term(spec, oracle_method(scheme=scheme, dynamics=dyn, brt=1), V)
    got = to_host(solver.term(ctx, spec, lib_method(scheme=scheme, dynamics=dyn, brt=1, kernel=1, tile=tile), to_dev(V)), n)
    assert np.isnan(want).any()
    if (scheme == 5 and np.isinf(mark)) or (scheme in (2, 3) and np.isnan(mark)):
        return
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
