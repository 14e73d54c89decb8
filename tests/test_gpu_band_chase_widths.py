"""Band reductions at widths that are no multiple of 4 (their columns do not suit
16-byte loads of FP32 operands), those over 128 in the general chase among
them, and the solves that go through such widths."""
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


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
@pytest.mark.parametrize("n,b,h", [(200, 33, 11), (150, 34, 17), (180, 45, 5), (120, 45, 9), (230, 50, 25), (300, 63, 21),
                                   (270, 66, 2), (300, 66, 22), (301, 70, 35), (260, 65, 13), (400, 110, 55), (390, 126, 63),
                                   (280, 127, 1), (500, 130, 10), (420, 140, 20), (67, 66, 33), (150, 75, 25)])
def test_widths(H, dtype_name, n, b, h):
    import torch

    dt = getattr(torch, dtype_name)
    A = I.random_band(n, b, 18000 + n + b + h)
    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b + n % 2).T)).to(dt).cuda()
    A = I.band_to_dense(AB.double().cpu().numpy().T)
    es = 8 if dtype_name == "float64" else 4
    if es * (3 * (b + 4) * h + (b + 4) * b + 3 * (h + 1) * h + h + 384) + 272 > 227 * 1024:
        # a chase's blocks do not fit one CTA's shared memory
        with pytest.raises(Exception, match="UNSUPPORTED"):
            H.band_to_band(AB, b, h)
        return
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > h] == 0.0)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS[dtype_name] * np.abs(lam).max()


@pytest.mark.parametrize("n,b0", [(150, 66), (67, 128), (200, 70), (130, 99), (260, 126), (103, 128)])
def test_solves_through_such_widths(H, n, b0):
    import torch

    A = I.semicircle(n, 18100 + n + b0)
    got = H.eigvalsh(torch.from_numpy(A).float().cuda(), b0).cpu().numpy()
    H.raise_device_error()
    lam = np.linalg.eigvalsh(A.astype(np.float32).astype(np.float64))
    assert np.abs(got - lam).max() <= 4 * n * EPS["float32"] * np.abs(lam).max() + 2e-9 * np.linalg.norm(A)
