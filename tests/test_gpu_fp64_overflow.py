"""FP64 element update without losses where the derivative's constant overflows: the clamp keeps the bound
that the infinite root lies beyond, as the oracle's division and clamp do."""
import numpy as np
import pytest

from paper_1903_10041_gb300 import workloads as W
from tests.test_gpu_parity import capi  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("y", [1e299, -1e299])
@pytest.mark.parametrize("n", [40, 40000])
def test_infinite_root_without_losses(capi, oracle_lib, n, y):  # noqa: F811
    P = W.random_problem(n, 1, 1, seed=60)
    P.g2[:], P.g1[:], P.g0[:], P.c[:], P.y[:] = 0.0, 0.0, 0.0, np.inf, y
    par = W.Params(rho=(1.0, 1.0 / n, 4e10, 1.0), max_iter=1, r_tol=0.0, s_tol=0.0)  # rho_3 y is infinite
    with capi.Solver(P, par) as s:
        s.solve(raise_on=())
        x = s.state()["x"]
    st, _ = oracle_lib.solve(P, par)
    want = P.hi if y > 0 else P.lo
    assert np.array_equal(st["x"][:, 0], want)
    assert np.array_equal(x[:, 0], want)
