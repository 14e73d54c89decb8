"""The batched kernel where its tiles end: orders around multiples of the 4 x 4
update tile, of the band and of the shared bisection levels (2^L - 1), strides
wider than the matrix, and the count of the shared levels bit for bit."""
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


SIZES = [2, 3, 4, 5, 6, 7, 8, 14, 15, 16, 17, 18, 31, 33, 34, 35, 63, 66, 127, 129, 190, 254, 255, 257]


@pytest.mark.parametrize("b,double", [(4, 0), (8, 0), (16, 0), (32, 0), (4, 1), (8, 1), (16, 1)])
def test_orders(H, b, double):
    """Backward stability of the reductions: eigenvalues within a few n eps of
    the exact ones, in units of ||A||_F, plus the bisection's tolerance."""
    import torch

    dt, eps, rtol = (torch.float64, 2.0**-52, 1e-14) if double else (torch.float32, 2.0**-23, 1e-9)
    host, dev = [], []
    for k, n in enumerate(SIZES):
        A = torch.from_numpy(I.semicircle(n, 15200 + k)).to(dt)
        wide = torch.full((n, n + k % 4), float("nan"), dtype=dt)
        wide[:, :n] = A
        host.append(A.double().numpy())
        dev.append(wide.cuda()[:, :n])
    got = [t.cpu().numpy() for t in H.eigvalsh_batched(dev, b)]
    H.raise_device_error()
    for A, lam in zip(host, got):
        n = A.shape[0]
        ref = np.linalg.eigvalsh(A)
        assert np.abs(lam - ref).max() <= (4 * n * eps + 2 * rtol) * np.linalg.norm(A), n


def test_tridiagonal_is_bisected_bitwise(H, orc):
    """An FP32 tridiagonal matrix passes through both reductions unchanged but
    for signs (a reflector of a single entry flips it, and the norm of one FP32
    entry is exact), so the result is the oracle's bisection of it."""
    import torch

    dev, ref = [], []
    for k, n in enumerate(SIZES):
        r = I.rng(15300 + k)
        d = r.standard_normal(n).astype(np.float32).astype(np.float64)
        e = r.standard_normal(n - 1).astype(np.float32).astype(np.float64)
        if k % 3 == 0:
            d[:] = 0.0  # the first midpoints hit exact zeros of the minors
        dev.append(torch.from_numpy(np.diag(d) + np.diag(e, 1) + np.diag(e, -1)).float().cuda())
        ref.append(orc.bisect(d, e, 1e-9))
    got = [t.cpu().numpy() for t in H.eigvalsh_batched(dev, 8)]
    H.raise_device_error()
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)
