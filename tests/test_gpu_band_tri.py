"""b -> 1 (the sliding-window kernel) where it can go wrong: several groups of
sweeps, a shared-memory ring that wraps, columns that the 16-byte copies cannot
serve (odd leading dimension), ragged ends, every supported width."""
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


def reduce_to_1(H, A, b, ldab, dtype):
    import torch

    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, ldab).T)).to(dtype).cuda()
    A32 = I.band_to_dense(AB.double().cpu().numpy().T)  # the matrix the GPU gets
    H.band_to_band(AB, b, 1)
    H.raise_device_error()
    return A32, I.band_to_dense(AB.double().cpu().numpy().T)


@pytest.mark.parametrize("n,b,pad", [(67, 2, 0), (130, 4, 0), (301, 8, 0), (301, 8, 1), (700, 16, 0), (699, 16, 3),
                                     (16, 16, 0), (17, 16, 0), (33, 16, 1), (34, 16, 0), (19, 2, 0), (21, 4, 1)])
def test_band_tri_fp64_vs_oracle(H, orc, n, b, pad):
    """Entry by entry: O(n u ||A||) per entry, the bound of the other band tests."""
    import torch

    A = I.random_band(n, min(b, n - 1), 13000 + n + b)
    A, got = reduce_to_1(H, A, b, 2 * b + pad, torch.float64)
    ref = orc.band_to_band(A, b, 1)
    np.testing.assert_allclose(np.tril(got), np.tril(ref), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > 1] == 0.0)


@pytest.mark.parametrize("n,b,pad", [(900, 2, 0), (900, 4, 0), (1100, 8, 0), (1100, 8, 1), (1300, 16, 0), (1301, 16, 2),
                                     (1500, 32, 0), (1499, 32, 1), (65, 32, 0), (33, 16, 0), (18, 4, 0)])
def test_band_tri_fp32_keeps_the_spectrum(H, n, b, pad):
    """The tridiagonal's eigenvalues against LAPACK's of the very band the GPU
    got.  n sweeps of backward stable similarities: ||E||_2 <= 4 n eps32 ||A||_2."""
    import torch

    A = I.random_band(n, b, 13100 + n + b)
    A, got = reduce_to_1(H, A, b, 2 * b + pad, torch.float32)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > 1] == 0.0)
