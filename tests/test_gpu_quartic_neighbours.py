"""The FP32 quartic kernel solves two elements at a time: an element's bits depend on its own data alone,
whatever stands beside it (invalid, A = 0, tied, undecided in FP32) and wherever it stands in the array."""
import numpy as np
import pytest

from tests.test_gpu_quartic import capi, quartics  # noqa: F401

pytestmark = pytest.mark.gpu


def solve(capi, a, bad=0):  # noqa: F811
    import torch
    d = [torch.from_numpy(v).cuda() for v in a]
    out = torch.empty_like(d[0])
    if bad:
        with pytest.raises(capi.AdmmError) as ei:
            capi.quartic_min(*d, precision="fp32", out=out)
        assert f"{bad} invalid" in str(ei.value)
    else:
        capi.quartic_min(*d, precision="fp32", out=out)
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 3, 200_001, 200_002])
def test_bits_do_not_depend_on_the_place(capi, n):  # noqa: F811
    a = [v.astype(np.float32) for v in quartics(n, seed=40)]
    x = solve(capi, a)
    pad = [np.concatenate([[v[0]], v]).astype(np.float32) for v in a]  # every element one place further
    assert np.array_equal(solve(capi, pad)[1:], x)


@pytest.mark.parametrize("kind", ["invalid", "quadratic", "tie", "triple"])
def test_bits_do_not_depend_on_the_neighbour(capi, kind):  # noqa: F811
    n = 200_000
    a = [v.astype(np.float32) for v in quartics(n, seed=41)]
    x = solve(capi, a)
    for start in (0, 1):
        b = [v.copy() for v in a]
        o = slice(start, None, 2)
        if kind == "invalid":
            b[0][o] = -1.0
        elif kind == "quadratic":
            b[0][o], b[2][o] = 0.0, 0.5
        elif kind == "tie":
            b[0][o], b[1][o], b[2][o], b[3][o] = 1.0, 0.0, -2.0, 0.0
        else:
            b[0][o] = 1.0
            b[1][o] = b[2][o] = b[3][o] = 0.0
        got = solve(capi, b, bad=n // 2 if kind == "invalid" else 0)
        assert np.array_equal(got[1 - start::2], x[1 - start::2])
