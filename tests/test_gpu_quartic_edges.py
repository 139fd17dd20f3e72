"""Quartic benchmark entry points at the edges: counts around pairs, blocks and the grid-stride loop, and
the inputs that leave the packed and seeded paths (exact ties, A = 0, tiny and huge coefficients, infinite
bounds, several minima outside the interval)."""
import numpy as np
import pytest

from tests.test_gpu_quartic import F, capi, quartics  # noqa: F401

pytestmark = pytest.mark.gpu

LOOP = 2 * 128 * 152 * 64  # elements at which the FP32 kernel starts taking several pairs per thread


@pytest.mark.parametrize("n", [1, 2, 3, 255, 256, 257, 513, LOOP - 1, LOOP + 3])
@pytest.mark.parametrize("mode", ["exact", "paper"])
def test_counts(capi, n, mode):  # noqa: F811
    """FP32 against FP64 on the same (FP32) inputs, by the value of the quartic: the bar of the FP32
    oracle test, and its share of positions (ties aside)."""
    import torch
    a = [torch.from_numpy(v).cuda() for v in quartics(n, seed=n)]
    x64 = capi.quartic_min(*a, mode=mode)
    x32 = capi.quartic_min(*[v.float() for v in a], mode=mode, precision="fp32").double()
    assert bool(torch.isfinite(x64).all()) and bool(torch.isfinite(x32).all())
    near = (x32 - x64).abs() <= 1e-4 * x64.abs().clamp(min=1.0)
    assert near.double().mean().item() > (0.999 if n > 1000 else 0.99)
    if mode == "exact":
        f64, f32 = F(*a[:4], x64), F(*a[:4], x32)
        assert bool((f32 <= f64 + 1e-5 * (1.0 + f64.abs())).all())


def special():
    rng = np.random.default_rng(3)
    n = 600
    A, B, C, D = rng.uniform(0.1, 2, n), rng.uniform(-2, 2, n), rng.uniform(-3, 3, n), rng.uniform(-2, 2, n)
    lo, hi = rng.uniform(-3, 0, n), rng.uniform(0, 3, n)
    k = np.arange(n)
    B[k % 12 == 0] = D[k % 12 == 0] = 0.0                                   # exact ties where C < 0
    lo[k % 12 == 1], hi[k % 12 == 1] = -np.inf, np.inf
    A[k % 12 == 2], C[k % 12 == 2] = 0.0, 0.5
    A[k % 12 == 3], C[k % 12 == 3] = 1e-35, 0.5                             # below the FP32 seeds' range
    for v in (A, B, C, D):
        v[k % 12 == 4] *= 1e35                                              # above it
    hi[k % 12 == 5] = lo[k % 12 == 5] = 0.25                                # a point
    lo[k % 12 == 6], hi[k % 12 == 6] = 5.0, 6.0                             # both minima left of the interval
    C[k % 12 == 7], lo[k % 12 == 7], hi[k % 12 == 7] = -3.0, -0.2, 0.2      # both minima outside, on both sides
    B[k % 12 == 8], C[k % 12 == 8], D[k % 12 == 8] = 0.0, 0.0, 0.0          # a triple root
    return A, B, C, D, lo, hi


@pytest.mark.parametrize("mode", ["exact", "paper"])
def test_fp64_special_inputs(capi, oracle_lib, mode):  # noqa: F811
    a = special()
    x, (xo, _) = capi.quartic_min(*a, mode=mode), oracle_lib.quartic_min(*a, mode=mode)
    A, B, C, D, lo, hi = a
    assert np.all((x >= lo) & (x <= hi))
    fg, fo = F(A, B, C, D, x), F(A, B, C, D, xo)
    scale = 1e-10 * (np.abs(A) + np.abs(B) + np.abs(C) + np.abs(D)) * (1.0 + np.abs(xo)) ** 4
    # A = 1e-35 goes to the closed form, as in the oracle, and both lose every digit of x there (b ~ 1e35)
    ok = np.arange(len(A)) % 12 != 3
    assert np.all((np.abs(fg - fo) <= scale)[ok]), np.argmax((np.abs(fg - fo) - scale)[ok])


def test_invalid_elements_are_counted_and_the_rest_solved(capi):  # noqa: F811
    import torch
    for prec, dt in (("fp64", torch.float64), ("fp32", torch.float32)):
        a = [torch.from_numpy(v).cuda().to(dt) for v in quartics(1001, seed=8)]
        good = capi.quartic_min(*a, precision=prec)
        bad = [v.clone() for v in a]
        bad[0][7], bad[1][8], bad[4][501], bad[3][1000] = -1.0, float("nan"), float("nan"), float("inf")
        bad[4][33], bad[5][33] = 1.0, 0.5
        out = torch.zeros_like(good)
        with pytest.raises(capi.AdmmError) as ei:
            capi.quartic_min(*bad, precision=prec, out=out)
        assert ei.value.status == capi.ADMM_EINVAL and "5 invalid" in str(ei.value)
        torch.cuda.synchronize()
        idx = [7, 8, 33, 501, 1000]
        assert bool(torch.isnan(out[idx]).all())
        keep = torch.ones(1001, dtype=torch.bool, device="cuda")
        keep[idx] = False
        assert torch.equal(out[keep], good[keep])
