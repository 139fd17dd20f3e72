"""The minimisers that the solve kernels run in step (a), on arrays (tests/solver_minimisers.cu): the FP32
pair minimiser of the mixed kernels and the factored FP64 element of the FP64 kernel, against the oracle's
Algorithm 1 and the exact golden cases.  The quartic entry points run variants of their own, so their tests
do not reach these."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from tests.test_gpu_quartic import F, quartics

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODE = {"exact": 0, "paper": 1}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_10041_gb300 import build
    so = str(tmp_path_factory.mktemp("minimisers") / "libsolver_minimisers.so")
    subprocess.run([build.NVCC, *build._flags(False), "-shared", "-o", so,
                    os.path.join(ROOT, "tests", "solver_minimisers.cu")], check=True)
    return C.CDLL(so)


def call(fn, arrays, *args):
    import torch
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
    x = torch.empty_like(d[0])
    torch.cuda.synchronize()
    assert fn(*[C.c_void_p(t.data_ptr()) for t in d], *args, C.c_void_p(x.data_ptr())) == 0
    return x.cpu().numpy().astype(np.float64)


def pairs(lib, a, mode="exact", tiny=False):
    a = [np.asarray(v, dtype=np.float32) for v in a]
    assert len(a[0]) % 2 == 0
    return call(lib.solver_pairs, a, len(a[0]) // 2, MODE[mode], int(tiny))


def elements(lib, b2, b1, u, Cc, Dh, hr1, lo, hi, mode="exact"):
    return call(lib.solver_elements, np.broadcast_arrays(b2, b1, u, Cc, Dh, hr1, lo, hi), len(b2), MODE[mode])


def expand(b2, b1, u, Cc, Dh, hr1):
    """A, B, C, D of Cc x^2 + 2 Dh x + hr1 (b2 x^2 + b1 x - u)^2."""
    return hr1 * b2 * b2, 2 * hr1 * b2 * b1, Cc + hr1 * (b1 * b1 - 2 * b2 * u), 2 * (Dh - hr1 * b1 * u)


def test_fp32_pairs_match_the_oracle(lib, oracle_lib):
    """The bars of the FP32 entry point's oracle test; a tenth of the pairs quadratic on both lanes."""
    a = quartics(200_000, seed=71)
    quad = np.zeros(200_000, dtype=bool)
    quad[:20_000] = True
    a[0][quad] = 0.0
    a[2][quad] = np.abs(a[2][quad]) + 0.125
    A, B, Cc, D, lo, hi = (v.astype(np.float32).astype(np.float64) for v in a)
    x_o, br = oracle_lib.quartic_min(A, B, Cc, D, lo, hi)
    assert all((br == t).mean() > 0.01 for t in (0, 2, 3))
    x = pairs(lib, (A, B, Cc, D, lo, hi))
    f_o, f = F(A, B, Cc, D, x_o), F(A, B, Cc, D, x)
    assert np.all(f <= f_o + 1e-5 * (1.0 + np.abs(f_o)))
    assert (np.abs(x - x_o) <= 1e-4 * np.maximum(1.0, np.abs(x_o))).mean() > 0.999


def test_fp32_pairs_whose_reciprocals_leave_the_range(lib, oracle_lib):
    from tests.test_gpu_quartic_fp32_special import special32
    a = special32()
    g = np.arange(len(a[0])) % 12
    low = (g >= 9) & (a[2] < 1e38)  # a huge C gives a zero quotient packed
    two = np.repeat(np.flatnonzero(low), 2)  # each such element on both lanes
    x = pairs(lib, [v[two] for v in a], tiny=True)
    xo, _ = oracle_lib.quartic_min(*[v[two].astype(np.float64) for v in a])
    assert np.all(np.abs(x - xo) <= 2.0 ** -23 * np.maximum(1.0, np.abs(xo)))


def golden():
    rows = [ln.split() for ln in open(os.path.join(ROOT, "tests", "golden", "quartic_cases.txt"))
            if not ln.startswith("#")]
    br = np.array([int(r[0]) for r in rows])
    v = np.array([[float(t) for t in r[1:]] for r in rows])
    return br, [np.ascontiguousarray(v[:, t]) for t in range(7)]


def test_fp32_pairs_meet_the_golden_cases(lib):
    """FP32 inputs are the rounded ones, so the bars are FP32's: the value to 1e-5 of its terms."""
    br, (A, B, Cc, D, lo, hi, want) = golden()
    if len(A) % 2:
        br, (A, B, Cc, D, lo, hi, want) = br[:-1], [v[:-1] for v in (A, B, Cc, D, lo, hi, want)]
    x = pairs(lib, (A, B, Cc, D, lo, hi))
    scale = (np.abs(A) + np.abs(B) + np.abs(Cc) + np.abs(D)) * (1.0 + np.abs(want)) ** 4
    assert np.all(F(A, B, Cc, D, x) <= F(A, B, Cc, D, want) + 1e-5 * scale)


def test_fp64_elements_meet_the_golden_cases(lib):
    """Each golden quartic (A > 0) in the factored form with hr1 = 1: b2 = sqrt(A), b1 = B / (2 b2), and u, Dh
    from C, D with a convex term K x^2.  Forming them rounds the coefficients by a few units of 2^-53 of
    their terms (K + b1^2 + |C| for C, |D| + |b1 u| for D): that is the slack of the value, and, where the
    minimum is not flat, of the position to 1e-9 as in the entry point's test."""
    br, (A, B, Cc, D, lo, hi, want) = golden()
    k = A > 0
    br, (A, B, Cc, D, lo, hi, want) = br[k], [v[k] for v in (A, B, Cc, D, lo, hi, want)]
    b2 = np.sqrt(A)
    b1 = B / (2 * b2)
    K = np.ones_like(A)
    u = (K + b1 * b1 - Cc) / (2 * b2)
    Dh = D / 2 + b1 * u
    x = elements(lib, b2, b1, u, K, Dh, np.ones_like(A), lo, hi)
    terms = K + b1 * b1 + np.abs(Cc) + np.abs(D) + np.abs(b1 * u) + A + np.abs(B)
    slack = 16 * np.finfo(float).eps * terms * (1.0 + np.abs(want)) ** 4
    f, fw = F(A, B, Cc, D, x), F(A, B, Cc, D, want)
    assert np.all(f <= fw + 1e-12 * (1.0 + np.abs(fw)) + slack)
    tie = (A == 1.0) & (B == 0.0) & (Cc == -2.0) & (D == 0.0)
    sure = (br != 1) & ~tie & (terms < 1e3)
    assert sure.sum() >= 50
    assert (np.abs(x - want) / np.maximum(1.0, np.abs(want)))[sure].max() <= 1e-9


@pytest.mark.parametrize("mode", ["exact", "paper"])
@pytest.mark.parametrize("kind", ["losses", "wells", "linear"])
def test_fp64_elements_match_the_oracle(lib, oracle_lib, mode, kind):
    """Coefficients as the solves meet them (losses), with two wells (large b2, u), and without losses: the
    bars of the FP64 entry point's oracle test."""
    n, rng = 100_001, np.random.default_rng(72)
    b2, b1 = rng.uniform(0.01, 0.1, n), rng.uniform(0.5, 1.5, n)
    u, Cc, Dh = rng.uniform(-2.0, 4.0, n), rng.uniform(0.25, 2.0, n), rng.uniform(-3.0, 3.0, n)
    lo, hi = rng.uniform(-3.0, 0.0, n), rng.uniform(0.0, 3.0, n)
    if kind == "wells":
        b2, b1, u = rng.uniform(0.3, 1.5, n), rng.uniform(-1.0, 1.0, n), rng.uniform(0.0, 8.0, n)
    if kind == "linear":
        b2[:] = b1[:] = 0.0
        b1[::3] = 0.5  # b2 = 0 alone: the quadratic case with losses
    hr1 = np.full(n, 0.5)
    A, B, C2, D = expand(b2, b1, u, Cc, Dh, hr1)
    x_o, br = oracle_lib.quartic_min(A, B, C2, D, lo, hi, mode=mode)
    if kind == "wells":
        assert (br == 2).mean() > 0.2
    x = elements(lib, b2, b1, u, Cc, Dh, hr1, lo, hi, mode)
    f_o, f = F(A, B, C2, D, x_o), F(A, B, C2, D, x)
    if mode == "exact":
        assert np.all(f <= f_o + 1e-10 * (1.0 + np.abs(f_o)))
    assert (np.abs(x - x_o) <= 1e-9 * np.maximum(1.0, np.abs(x_o))).mean() > 0.9999
