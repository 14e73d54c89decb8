"""Bisection, bit for bit against the oracle's restatement of the recurrence, at
the edges of the Sturm count's blocks, on both sides of the order where the
rounds keep their state in shared memory, and on matrices whose minors vanish,
shrink by hundreds of binades or meet underflowing squares."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def matrix(kind, n):
    r = I.rng(13700 + n)
    d, e = r.standard_normal(n), r.standard_normal(max(n - 1, 0))
    if kind == "identity":
        d, e = np.ones(n), np.zeros(n - 1)
    elif kind == "blocks":  # exact zeros off the diagonal, repeated diagonal entries
        d = np.repeat(r.standard_normal(n), 1 + (np.arange(n) % 3))[:n]
        e[np.arange(n - 1) % 5 == 0] = 0.0
    elif kind == "zero_diagonal":  # midpoint 0: every other minor vanishes
        d = np.zeros(n)
        e = np.ones(n - 1)
    elif kind == "graded":
        g = 10.0 ** np.linspace(0, -90, n)
        d, e = d * g, e * g[1:]
    elif kind == "tiny_e":  # squares underflow
        e = e * 10.0 ** r.integers(-200, 1, n - 1)
    return d, e


@pytest.mark.parametrize("n", [2, 3, 8, 9, 10, 16, 17, 18, 25, 33])
def test_block_edges(H, orc, n):
    import torch

    d, e = matrix("random", n)
    for rtol in (1e-9, 1e-14):
        got = H.tridiag_bisect(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda(), rtol).cpu().numpy()
        H.raise_device_error()
        np.testing.assert_array_equal(got, orc.bisect(d, e, rtol))


@pytest.mark.parametrize("n", [300, 2047, 2048, 2049])
@pytest.mark.parametrize("kind", ["random", "identity", "blocks", "zero_diagonal", "graded", "tiny_e"])
def test_special_matrices(H, orc, kind, n):
    import torch

    if n > 300 and kind in ("identity", "tiny_e") and n != 2049:
        pytest.skip("one order past the small kernel is enough")
    d, e = matrix(kind, n)
    got = H.tridiag_bisect(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda(), 1e-14).cpu().numpy()
    H.raise_device_error()
    np.testing.assert_array_equal(got, orc.bisect(d, e, 1e-14))
