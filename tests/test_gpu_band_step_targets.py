"""The step kernel at targets that are no multiple of the columns it reads at once
(2 over a width of 32, 4 over 64), at its widest targets, and where its shared
memory is nearly full."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = {"float32": 2.0**-23, "float64": 2.0**-52}


@pytest.fixture(scope="module")
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


SHAPES = [(150, 33, 1), (171, 33, 11), (200, 45, 5), (200, 45, 15), (140, 48, 3), (97, 63, 7), (260, 63, 21), (200, 64, 1),
          (300, 66, 1), (301, 66, 2), (290, 66, 11), (303, 66, 22), (280, 72, 9), (290, 96, 6), (321, 96, 32), (350, 100, 25),
          (400, 120, 24), (300, 112, 28), (310, 112, 7), (300, 127, 1), (390, 128, 1), (400, 128, 2), (131, 128, 2)]


@pytest.mark.parametrize("n,b,h", SHAPES)
def test_fp64_vs_oracle(H, orc, n, b, h):
    """Entry by entry: O(n u ||A||), the bound of the other band tests."""
    import torch

    A = I.random_band(n, b, 18200 + n + b + h)
    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b + n % 2).T)).cuda()
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    got = I.band_to_dense(AB.cpu().numpy().T)
    ref = orc.band_to_band(A, b, h)
    np.testing.assert_allclose(np.tril(got), np.tril(ref), atol=20 * n * EPS["float64"] * np.linalg.norm(A), rtol=0)
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > h] == 0.0)


@pytest.mark.parametrize("n,b,h", SHAPES + [(500, 128, 64), (193, 128, 64), (400, 126, 63), (370, 120, 60), (260, 70, 35),
                                            (900, 50, 25), (700, 54, 27), (600, 60, 15)])
def test_fp32_keeps_the_spectrum(H, n, b, h):
    """Backward stable similarities: ||E||_2 <= 4 n eps32 ||A||_2."""
    import torch

    A = I.random_band(n, b, 18300 + n + b + h)
    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b + n % 2).T)).float().cuda()
    A = I.band_to_dense(AB.double().cpu().numpy().T)
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS["float32"] * np.abs(lam).max()
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > h] == 0.0)
