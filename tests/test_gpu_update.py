"""The products of the trailing update where they can go wrong: unaligned FP32
matrices (reduced in an aligned copy, or in place when there is no room for
one), split products at sizes off every tile, both tile widths."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS64 = np.finfo(np.float64).eps
EPS32 = float(np.finfo(np.float32).eps)


@pytest.fixture(scope="module")
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def strided(A, ld, shift=0):
    """A as an n x n float32 CUDA tensor with row stride ld, starting `shift` elements into its buffer."""
    import torch

    n = A.shape[0]
    buf = torch.full((n * ld + shift,), float("nan"), dtype=torch.float32, device="cuda")
    t = buf[shift:].view(n, ld)[:, :n]
    t.copy_(torch.from_numpy(A).float())
    return t


@pytest.mark.parametrize("n,b,ld,shift", [(1101, 64, 1101, 0), (1102, 64, 1103, 0), (1100, 32, 1100, 1), (1103, 128, 1103, 3),
                                          (900, 24, 901, 0)])
def test_unaligned_matrix(H, n, b, ld, shift):
    """Reduced in an aligned copy: the band's spectrum (FP32 products throughout:
    ||E||_2 <= n eps32 ||A||_2), and A holds the band as documented."""
    A = I.semicircle(n, 14300 + n + b).astype(np.float32).astype(np.float64)
    ut = strided(A, ld, shift)
    AB = H.full_to_band(ut, b)
    H.raise_device_error()
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= n * EPS32 * np.abs(lam).max()
    # the band, exact zeros below it (the transpose of the lower triangle, row-major)
    np.testing.assert_array_equal(np.triu(ut.double().cpu().numpy()).T, np.tril(got))


def test_unaligned_matrix_in_a_workspace_of_the_queried_size(H):
    """No room for the copy: the reduction runs on the matrix as it is."""
    import torch

    n, b0 = 1101, 64
    A = I.semicircle(n, 14400)
    lam = np.linalg.eigvalsh(A)
    ws = torch.empty(H.workspace_query(n, b0, 1), dtype=torch.uint8, device="cuda")
    H.set_workspace(ws)
    try:
        got = H.eigvalsh(strided(A, n), b0).cpu().numpy()
        H.raise_device_error()
    finally:
        H.set_workspace(None)
    again = H.eigvalsh(strided(A, n), b0).cpu().numpy()
    H.raise_device_error()
    for g in (got, again):
        assert np.abs(g - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()


@pytest.mark.parametrize("n,b", [(1000, 32), (777, 64), (1000, 16), (515, 33), (2100, 64)])
def test_fp64_split_products_keep_the_spectrum(H, n, b):
    import torch

    A = I.semicircle(n, 14500 + n + b)
    AB = H.full_to_band(torch.from_numpy(A).cuda(), b)
    H.raise_device_error()
    got = I.band_to_dense(AB.cpu().numpy().T)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS64 * np.abs(lam).max()


@pytest.mark.parametrize("n,b", [(1500, 128), (900, 96), (700, 31), (2051, 64), (400, 7)])
def test_fp32_products_keep_the_spectrum(H, n, b):
    import torch

    A = I.semicircle(n, 14600 + n + b)
    AB = H.full_to_band(torch.from_numpy(A).float().cuda(), b)
    H.raise_device_error()
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    lam = np.linalg.eigvalsh(A.astype(np.float32).astype(np.float64))
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()
