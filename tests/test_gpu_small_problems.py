"""Single instances around the sizes where the launch shape changes (one CTA, one cluster, the whole
grid; a piece of one row per CTA), and elements on every branch of the FP64 update, against the FP64
oracle.  FP64 to 1e-9 of the state (the bar of the parity tests); mixed precision after five iterations
to 1e-5 (the bar of its trajectory test)."""
import numpy as np
import pytest

from paper_1903_10041_gb300 import workloads as W
from tests.test_gpu_parity import capi, compare_states, double_well, run_both  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (31, 2, 1), (128, 2, 1), (129, 3, 1), (1024, 2, 1), (1025, 2, 1), (30, 8, 8), (30, 5, 9),
         (100, 1, 8), (257, 4, 2), (500, 2, 3)]


@pytest.mark.parametrize("n,m,q", SIZES)
@pytest.mark.parametrize("adapt", [False, True])
def test_fp64_small_sizes(capi, oracle_lib, n, m, q, adapt):  # noqa: F811
    P = W.random_problem(n, m, q, seed=1000 + n)
    par = W.Params(rho=(1.0, 1.0 / n, 1.0, 1.0), max_iter=45, r_tol=0.0 if not adapt else 1e-12,
                   s_tol=0.0 if not adapt else 1e-12, adapt_rho=adapt)
    compare_states(P, *run_both(capi, oracle_lib, P, par))


@pytest.mark.parametrize("n,m,q", [(1, 1, 1), (129, 2, 1), (512, 4, 1), (513, 4, 1), (4096, 2, 1), (4097, 2, 1),
                                   (60, 6, 8), (60, 3, 9)])
def test_mixed_small_sizes_track_the_oracle(capi, oracle_lib, n, m, q):  # noqa: F811
    P = W.random_problem(n, m, q, seed=2000 + n)
    par = W.Params(rho=(1.0, 1.0 / n, 1.0, 1.0), max_iter=5, r_tol=0.0, s_tol=0.0)
    st_o, _ = oracle_lib.solve(P, par)
    with capi.Solver(P, par.replace(precision="mixed")) as s:
        s.solve(raise_on=(1, 2, 3, 4, 6))
        st = s.state()
    assert np.abs(st["x"] - st_o["x"]).max() <= 1e-5 * max(1.0, np.abs(st_o["x"]).max())


def branches():
    """Sources on every branch: two wells inside wide bounds, two wells with an interval on one side,
    linear losses (g2 = 0), no losses, tiny g2, and a g2 below the FP32 range."""
    P = double_well(130, 6, 3, seed=5)
    P.lo[0], P.hi[0] = -4.0, 4.0
    P.lo[1], P.hi[1] = 0.75, 4.0
    P.g2[2] = 0.0
    P.g2[3], P.g1[3], P.g0[3] = 0.0, 0.0, 0.0
    P.g2[4] = 1e-6
    P.g2[5], P.g1[5] = 1e-200, np.abs(P.g1[5]) + 0.5
    return P


@pytest.mark.parametrize("mode", ["exact", "paper"])
@pytest.mark.parametrize("sweep", ["gauss_seidel", "jacobi"])
@pytest.mark.parametrize("tiny,iters", [(1e-6, 1), (0.5, 25)])
def test_fp64_branches_of_the_element_update(capi, oracle_lib, mode, sweep, tiny, iters):  # noqa: F811
    """Against the oracle: one iteration with the tiny g2, whose closed form in the oracle is itself
    3.8e-10 off (next test) and drifts above the bar in later iterations; 25 without it."""
    P = branches()
    P.g2[4] = tiny
    par = W.Params(max_iter=iters, r_tol=0.0, s_tol=0.0, xmin_mode=mode, sweep=sweep)
    compare_states(P, *run_both(capi, oracle_lib, P, par), check_res=iters > 1)


def test_fp64_tiny_losses_against_long_double(capi):  # noqa: F811
    """Step (a) of the first iteration (Jacobi, from zeros) for the convex sources, by Newton in long
    double: within a few ulp, tiny g2 included (where the closed form loses half the digits)."""
    P = branches()
    m, q, n, L = P.m, P.q, P.n, np.longdouble
    with capi.Solver(P, W.Params(max_iter=1, r_tol=0.0, s_tol=0.0, sweep="jacobi")) as s:
        s.solve(raise_on=(1, 2, 3, 4, 6))
        got = s.state()["x"]
    x0 = np.clip(0.0, P.lo, P.hi)[:, None, :] * np.ones((m, q, n))
    for i in (2, 4, 5):
        phi = P.y - (x0.sum(0) - x0[i])
        a2, a1, b2, b1, u = (v[i].astype(L) for v in (P.f2, P.f1, P.g2, P.g1, -P.g0))
        C, Dh = a2 / q + L(0.5), (a1 / q - phi) / 2
        C[:, 0] += L(0.5)
        x = -(Dh - b1 * u / 2) / (C + b1 * b1 / 2)
        for _ in range(30):
            e, gp = (b2 * x + b1) * x - u, 2 * b2 * x + b1
            x = x - (C * x + Dh + e * gp / 2) / (C + (gp * gp + 2 * b2 * e) / 2)
        want = np.clip(x, P.lo[i], P.hi[i]).astype(float)
        assert np.abs(got[i] - want).max() <= 16 * np.finfo(float).eps * max(1.0, np.abs(want).max()), i
