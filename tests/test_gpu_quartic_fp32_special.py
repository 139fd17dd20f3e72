"""The FP32 quartic entry point on the special inputs of the FP64 edge test, with groups whose reciprocals
leave the FP32 range: A = 0 with a denormal or huge C, and a denormal A at a triple root."""
import numpy as np
import pytest

from tests.test_gpu_quartic import F, capi  # noqa: F401
from tests.test_gpu_quartic_edges import special

pytestmark = pytest.mark.gpu


def special32():
    A, B, C, D, lo, hi = special()
    k = np.arange(len(A))
    g, t = k % 12, k // 12 % 3
    tiny = 2.0 ** -127
    sign = np.array([1.0, -1.0, 0.0])[t]
    for v in (A, B, C, D):
        v[g >= 9] = 0.0
    lo[g >= 9], hi[g >= 9] = -1.0, 1.0
    C[g == 9], D[g == 9] = 4e-39, 1e-39 * sign[g == 9]                       # x = -D / (2 C), 2 C denormal
    A[g == 10], B[g == 10], C[g == 10], D[g == 10] = tiny, -4 * tiny, 6 * tiny, -4 * tiny  # tiny (x - 1)^4
    lo[g == 10], hi[g == 10] = -3.0, 3.0
    A[g == 11] = tiny                                                        # tiny x^4
    big = (g == 11) & (t == 1)
    A[big], C[big], D[big] = 0.0, 1.5e38, -1e38                              # 1 / (2 C) denormal
    return [v.astype(np.float32) for v in (A, B, C, D, lo, hi)]


@pytest.mark.parametrize("mode", ["exact", "paper"])
def test_fp32_special_inputs(capi, oracle_lib, mode):  # noqa: F811
    """Groups 9 to 11 have one minimum and FP64 room: FP32 rounding of the oracle's x.  The others by the
    value of the quartic, the bar of the FP32 oracle test scaled by the terms; group 3 (A = 1e-35) has no
    digits in either closed form, and the literal Pi(argmin) of a near tie is either clamped root."""
    a = special32()
    x = capi.quartic_min(*a, mode=mode, precision="fp32").astype(np.float64)
    A, B, C, D, lo, hi = (v.astype(np.float64) for v in a)
    xo, _ = oracle_lib.quartic_min(A, B, C, D, lo, hi, mode=mode)
    g = np.arange(len(A)) % 12
    assert np.all((x >= lo) & (x <= hi)), g[~((x >= lo) & (x <= hi))]
    far = (g >= 9) & ~(np.abs(x - xo) <= 2.0 ** -23 * np.maximum(1.0, np.abs(xo)))
    assert not far.any(), (g[far], x[far], xo[far])
    if mode == "exact":
        scale = 1e-5 * (np.abs(A) + np.abs(B) + np.abs(C) + np.abs(D)) * (1.0 + np.abs(xo)) ** 4
        ok = (g != 3) & (g < 9)
        assert np.all((np.abs(F(A, B, C, D, x) - F(A, B, C, D, xo)) <= scale)[ok])


@pytest.mark.parametrize("m,batch", [(1, False), (6, False), (1, True), (6, True)])
def test_mixed_solves_with_a_denormal_rho3(capi, m, batch):  # noqa: F811
    """Step (a) of the first iteration without costs and losses: x = s - others + y + mu, the quotient of two
    denormal numbers in FP32 (about 22 bits each)."""
    from paper_1903_10041_gb300 import workloads as W
    n, q = 301, 2
    P = W.random_problem(n, m, q, seed=90)
    for v in (P.f2, P.f1, P.g2, P.g1, P.g0):
        v[:] = 0.0
    P.c[:], P.lo[:], P.hi[:] = np.inf, 0.0, 4.0
    par = W.Params(rho=(1.0, 1.0 / n, 6e-39, 1.0), max_iter=1, r_tol=0.0, s_tol=0.0, precision="mixed")
    if batch:
        with capi.Batch([P], par) as b:
            b.solve()
            b.wait()
            x = b.state(0)["x"]
    else:
        with capi.Solver(P, par) as s:
            s.solve(raise_on=())
            x = s.state()["x"]
    assert np.abs(x[0, :, 1:] - P.y[:, 1:]).max() <= 1e-5
    assert np.abs(x[1:, :, 1:]).max(initial=0.0) <= 1e-5  # the first source has taken the demand
