"""Results of a batch in device buffers (one launch) against the same results in host buffers, and the
zero start set on the device against a new batch's, at the smallest and ragged sizes."""
import ctypes

import numpy as np
import pytest

from paper_1903_10041_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_10041_gb300 import build
    build.build()
    from paper_1903_10041_gb300 import capi
    return capi


@pytest.mark.parametrize("shapes", [[(1, 1, 1)], [(2, 1, 3), (37, 3, 5), (64, 2, 1), (1029, 4, 7)],
                                    [(50, 8, 2), (33, 2, 31)]])
def test_device_results_equal_host_results(capi, shapes):
    import torch
    P = [W.random_problem(n, m, q, seed=100 + t) for t, (n, m, q) in enumerate(shapes)]
    par = W.Params(rho2_over_n=True, precision="mixed", max_iter=30)
    dp = ctypes.POINTER(ctypes.c_double)
    with capi.Batch(P, par) as b:
        b.solve()
        host = b.wait(want_x=True)
        x = [torch.full((m * q * n + 1,), 7.0, dtype=torch.float64, device="cuda") for n, m, q in shapes]
        x1 = [torch.full((m + 1,), 7.0, dtype=torch.float64, device="cuda") for n, m, q in shapes]
        res = (capi.admm_result * len(P))()
        for t, r in enumerate(res):
            r.x = ctypes.cast(ctypes.c_void_p(x[t].data_ptr()), dp)
            if t % 2 == 0:  # x alone for every second instance
                r.x1 = ctypes.cast(ctypes.c_void_p(x1[t].data_ptr()), dp)
            r.on_device = 1
        st = capi._lib.admm_batch_wait(b.h, None, res)
        assert st in (capi.ADMM_OK, capi.ADMM_ENOTCONVERGED)
        for t, (n, m, q) in enumerate(shapes):
            xt, x1t = x[t].cpu().numpy(), x1[t].cpu().numpy()
            assert np.array_equal(xt[:-1].reshape(m, q, n), host[t]["x"]) and xt[-1] == 7.0
            assert np.array_equal(x1t[:-1], host[t]["x1"]) if t % 2 == 0 else np.all(x1t == 7.0)
            assert x1t[-1] == 7.0
        # the zero start set on the device gives a new batch's state and solve
        b.reset()
        with capi.Batch(P, par) as fresh:
            for t in range(len(P)):
                s0, s1 = b.state(t), fresh.state(t)
                for k in s0:
                    assert np.array_equal(s0[k], s1[k]), k
        b.solve()
        again = b.wait(want_x=True)
        for t in range(len(P)):
            assert np.array_equal(again[t]["x"], host[t]["x"]) and again[t]["iters"] == host[t]["iters"]


@pytest.mark.parametrize("cfg", [(16, 0, 0, 1, 0), (8, 0, 4096, 1, 0), (8, 0, 0, 2, 2048)])
def test_a_batch_resumed_anywhere_gives_the_same_bits(capi, cfg):
    """A solve cut at any iteration (a check there, where the whole run has none) and continued from its
    saved state takes the whole run's bits: check and plain iterations round alike, and the scalar state
    read back gives the same FP32 offsets as the one kept on chip (ties among them: q = 2 means)."""
    shapes = [(276, 4, 18), (139, 4, 6), (600, 2, 2), (77, 3, 2), (33, 1, 1)]
    P = [W.random_problem(n, m, q, seed=300 + t) for t, (n, m, q) in enumerate(shapes)]

    def run(iters, states=None):
        par = W.Params(rho=(1.0, 1.0 / 600, 1.0, 1.0), precision="mixed", max_iter=iters)
        with capi.Batch(P, par) as b:
            b.set_config(*cfg)
            for t, s in enumerate(states or []):
                b.set_state(t, s)
            b.solve()
            b.wait()
            return [b.state(t) for t in range(len(P))]

    whole = run(47)
    for cut in (1, 10, 23):
        part = run(47 - cut, run(cut))
        for t in range(len(P)):
            for k in whole[t]:
                assert np.array_equal(whole[t][k], part[t][k]), (cut, t, k)


@pytest.mark.parametrize("precision,n,m,q", [("mixed", 600, 2, 2), ("mixed", 2003, 4, 6), ("mixed", 301, 6, 3),
                                             ("fp64", 301, 3, 2)])
def test_a_single_solve_resumed_anywhere_gives_the_same_bits(capi, precision, n, m, q):
    P = W.random_problem(n, m, q, seed=77)

    def run(iters, warm=None):
        par = W.Params(rho=(1.0, 1.0 / n, 1.0, 1.0), precision=precision, max_iter=iters)
        with capi.Solver(P, par) as s:
            s.solve(warm=warm)
            return s.state()

    whole = run(47)
    for cut in (1, 10, 23):
        part = run(47 - cut, run(cut))
        for k in whole:
            assert np.array_equal(whole[k], part[k]), (cut, k)


def test_device_results_in_any_kind_of_buffer(capi):
    """Neighbouring ranges of one allocation, NULL, and a misaligned buffer that takes the copies, in one call."""
    import torch
    shapes = [(37, 3, 5), (64, 2, 1), (50, 2, 2), (33, 4, 3)]
    P = [W.random_problem(n, m, q, seed=400 + t) for t, (n, m, q) in enumerate(shapes)]
    dp = ctypes.POINTER(ctypes.c_double)
    with capi.Batch(P, W.Params(rho2_over_n=True, precision="mixed", max_iter=20)) as b:
        b.solve()
        host = b.wait(want_x=True)
        size = [n * m * q for n, m, q in shapes]
        one = torch.full((sum(size) * 8 + 4,), 7, dtype=torch.uint8, device="cuda")
        res = (capi.admm_result * len(P))()
        at = [0]
        for t, r in enumerate(res):
            off = 8 * at[-1] + (4 if t == 3 else 0)  # the last one misaligned
            r.x = ctypes.cast(ctypes.c_void_p(one.data_ptr() + off), dp) if t != 1 else None
            r.on_device = 1
            at.append(at[-1] + size[t])
        assert capi._lib.admm_batch_wait(b.h, None, res) in (capi.ADMM_OK, capi.ADMM_ENOTCONVERGED)
        got = one.cpu().numpy()
        for t, (n, m, q) in enumerate(shapes):
            off = 8 * at[t] + (4 if t == 3 else 0)
            raw = got[off:off + 8 * size[t]]
            if t == 1:
                assert np.all(raw == 7)
            else:
                assert np.array_equal(raw.copy().view(np.float64).reshape(m, q, n), host[t]["x"])


@pytest.mark.parametrize("n,m,q", [(40, 2, 54), (33, 1, 108)])
def test_shapes_that_just_fit_a_cta_of_16_warp_teams(capi, n, m, q):
    """Sixteen one-warp teams side by side need nearly all of an SM's shared memory at these shapes; the bits
    are those of four in a CTA."""
    P = [W.random_problem(n, m, q, seed=500 + t) for t in range(20)]
    x = []
    for warps in (4, 16):
        with capi.Batch(P, W.Params(rho2_over_n=True, precision="mixed", max_iter=25)) as b:
            b.set_config(warps, 0, 1 << 20, 1, 1 << 20)
            b.solve()
            x.append([r["x"] for r in b.wait(want_x=True)])
    assert all(np.array_equal(u, v) for u, v in zip(*x))
