"""hj_upwind beyond the parity fields: FP32 data of any size."""
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
