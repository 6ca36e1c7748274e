"""hj_upwind beyond the parity fields: FP32 data of any size, FP32 lines of
dimension 0 (interfaces dealt out two a thread, whatever the lines) at the sizes
where the deal can go wrong, and what dimension 0 costs beside the others."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_11542_gb300 import workloads as W
from helpers import NORM, lib_method, oracle_method, rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11542_gb300 import solver
    with solver.Context(0) as c:
        yield c


@pytest.mark.parametrize("size", [1.0, 4e8, 1e12, 1e19, 1e30, 3e36])
@pytest.mark.parametrize("dim", [0, 1, 2])
def test_fp32_weno5_of_any_size(ctx, size, dim):
    """The squared smoothness sums of FP32 data leave FP32 from differences of
    about 1e9 on; the derivatives do not. White noise, so that no window is
    smooth; each result a sum of a few rounded terms of the data's size (2^-24
    each, amplified by the weights' sensitivity: the parity tests' 2e-4)."""
    from paper_2507_11542_gb300 import solver
    spec = W.GridSpec((45, 17, 11), (-1.0, 0.0, 0.0), (2.0, 1.0, 6.0), (2,))
    V = np.random.default_rng(8).uniform(-size, size, spec.n)
    V32 = np.asfortranarray(np.float32(V).astype(np.float64))
    pm_o, pp_o = O.upwind(spec, oracle_method(dynamics=NORM), V32, dim)
    pm, pp = solver.upwind(ctx, spec, lib_method(dynamics=NORM), to_dev(V32, "float32"), dim)
    for got, want in ((pm, pm_o), (pp, pp_o)):
        got = to_host(got, spec.n)
        assert np.isfinite(got).all()
        assert rel_err(got, want) < 2e-4


@pytest.mark.parametrize("n,periodic", [((1, 6), (0,)), ((2,), ()), ((3, 3), ()), ((4, 1), (1,)), ((127,), ()), ((128,), (0,)),
                                        ((5, 7, 3), (0, 1)), ((6, 1, 1), (1, 2)), ((255, 3), (1,)), ((1, 1, 300), (0, 1))])
@pytest.mark.parametrize("scheme", [1, 2, 3, 5])
@pytest.mark.parametrize("extrap", [0, 1])
def test_fp32_lines_of_stride_one(ctx, n, periodic, scheme, extrap):
    """Odd and even numbers of interfaces, lines shorter than the stencil, one
    line, a dimension of stride 1 behind dimensions of one node. Rounding of
    data of size 1 over dx: the parity tests' 2e-4."""
    from paper_2507_11542_gb300 import solver
    spec = W.GridSpec(n, (-1.0, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0)[:len(n)], periodic)
    V = np.random.default_rng(5).uniform(-1.0, 1.0, n)
    V32 = np.asfortranarray(np.float32(V).astype(np.float64))
    for dim in range(len(n)):
        pm_o, pp_o = O.upwind(spec, oracle_method(scheme=scheme, dynamics=NORM, extrap=extrap), V32, dim)
        pm, pp = solver.upwind(ctx, spec, lib_method(scheme=scheme, dynamics=NORM, extrap=extrap), to_dev(V32, "float32"), dim)
        assert rel_err(to_host(pm, n), pm_o) < 2e-4
        assert rel_err(to_host(pp, n), pp_o) < 2e-4


def test_fp32_dimension_0_costs_what_the_others_do(ctx):
    """The same bytes along every dimension of 300^3 (27 M nodes, far larger than
    a launch's cost): dimension 0 may take twice the last dimension's time, where
    a thread that runs along the line takes three times."""
    import torch
    from paper_2507_11542_gb300 import solver
    spec = W.GridSpec((300, 300, 300), (-1.0,) * 3, (1.0,) * 3)
    V = torch.rand(27000000, device="cuda")
    m = lib_method(scheme=1, dynamics=NORM)

    def best(dim):
        took = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                solver.upwind(ctx, spec, m, V, dim)
            b.record()
            torch.cuda.synchronize()
            took.append(a.elapsed_time(b))
        return min(took)

    best(2)
    assert best(0) <= 2.0 * best(2)
