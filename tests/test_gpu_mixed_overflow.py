"""Mixed precision takes FP64-finite data that overflow in FP32.  The NaN or infinity that a column then
holds stays one in the row sums and residuals, as the FP64 conversions would keep it, and the solve does
not pass its stop test."""
import numpy as np
import pytest

from paper_1903_10041_gb300 import workloads as W
from tests.test_gpu_parity import capi  # noqa: F401

pytestmark = pytest.mark.gpu

CONFIGS = [(16, 0, 0, 1, 0), (8, 0, 0, 1, 0), (8, 0, 1 << 20, 1, 1 << 20), (8, 0, 0, 2, 0)]  # CTA, warp, cluster teams
PAR = dict(rho2_over_n=True, precision="mixed", max_iter=3000)


def overflowing(n, m, q, k, array="f2"):
    """f2: x of the column is NaN after one iteration.  y: a demand no x meets, infinite in FP32.  With a
    capacity of +inf h follows 1'z, so a finite constant in the place of a NaN sum would settle."""
    P = W.random_problem(n, m, q, seed=50 + n)
    P.c[:] = np.inf
    if array == "f2":
        P.f2[0, 0, k] = 1e39
    else:
        P.y[0, k] = 1e39
    return P


def check_first_iteration(st, k):
    assert np.isnan(st["x"][0, 0, k])
    gone = np.isnan(st["x"]).any(axis=2)
    assert np.all(np.isnan(st["lam"][gone])) and np.all(np.isfinite(st["lam"][~gone]))
    if k == 0:
        assert np.isnan(st["x1"][0])


@pytest.mark.parametrize("k", [0, 3])
@pytest.mark.parametrize("n,m,q", [(300, 2, 1), (3000, 3, 6), (600, 6, 2), (2000, 6, 5)])
def test_single(capi, n, m, q, k):  # noqa: F811
    """One cluster and the grid, m <= 4 and above."""
    with capi.Solver(overflowing(n, m, q, k), W.Params(**dict(PAR, max_iter=1))) as s:
        s.solve(raise_on=())
        check_first_iteration(s.state(), k)
    for array in ("f2", "y"):
        with capi.Solver(overflowing(n, m, q, k, array), W.Params(**PAR)) as s:
            r = s.solve(raise_on=())
        assert not r["converged"] and r["iters"] == 3000, array


@pytest.mark.parametrize("k", [0, 3])
@pytest.mark.parametrize("cfg", CONFIGS)
def test_batch(capi, cfg, k):  # noqa: F811
    """m <= 4 and above; a sound instance beside the others converges."""
    small = [(300, 2, 1), (500, 4, 3), (400, 2, 2)]
    for shapes in (small, [(n, m + 4, q) for n, m, q in small]):
        P = [overflowing(*shapes[0], k), overflowing(*shapes[1], k), overflowing(*shapes[1], k, "y"),
             W.random_problem(*shapes[2], seed=9)]
        for iters in (1, 3000):
            with capi.Batch(P, W.Params(**dict(PAR, max_iter=iters))) as b:
                b.set_config(*cfg)
                b.solve()
                r = b.wait()
                if iters == 1:
                    check_first_iteration(b.state(0), k)
                    check_first_iteration(b.state(1), k)
                    continue
            assert not any(r[t]["converged"] for t in (0, 1, 2)), [r[t]["converged"] for t in (0, 1, 2)]
            assert r[3]["converged"]
