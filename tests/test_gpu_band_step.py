"""The band step kernel (b -> h, h > 1) where it can go wrong: widths that are no
multiple of 4, targets below a tile, ragged last blocks of every length, one
and several CTAs per sweep, the last steps of a sweep with one or no row below."""
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


def reduce(H, A, b, h, dtype, pad=0):
    import torch

    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b + pad).T)).to(dtype).cuda()
    A = I.band_to_dense(AB.double().cpu().numpy().T)  # the matrix the GPU gets
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > h] == 0.0)
    return A, got


CASES64 = [(130, 4, 2), (131, 8, 2), (97, 8, 4), (150, 6, 3), (100, 9, 3), (77, 12, 4), (203, 16, 8), (161, 32, 16),
           (170, 32, 4), (33, 32, 16), (34, 32, 16), (65, 32, 16), (66, 32, 8), (301, 64, 16), (129, 64, 32),
           (193, 64, 2), (300, 96, 32), (385, 128, 16), (400, 128, 8), (60, 20, 10),
           (400, 4, 2), (620, 4, 2)]  # (more sweeps at once than one CTA per SM)


@pytest.mark.parametrize("n,b,h", CASES64)
def test_band_step_fp64_vs_oracle(H, orc, n, b, h):
    import torch

    A = I.random_band(n, b, 13800 + n + b + h)
    A, got = reduce(H, A, b, h, torch.float64, pad=n % 2)
    ref = orc.band_to_band(A, b, h)
    np.testing.assert_allclose(np.tril(got), np.tril(ref), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)


def test_band_step_fp64_one_cta_per_sm(H):
    """A wide FP64 band whose sweeps are limited to one CTA per SM."""
    import torch

    n, b, h = 2400, 32, 16
    A = I.random_band(n, b, 13850)
    A, got = reduce(H, A, b, h, torch.float64)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 20 * n * EPS64 * np.abs(lam).max()


@pytest.mark.parametrize("n,b,h", [(900, 32, 16), (901, 32, 8), (700, 64, 16), (701, 64, 8), (515, 128, 32), (513, 128, 64),
                                   (400, 24, 6), (300, 10, 5), (257, 128, 4), (300, 16, 2), (200, 100, 20)])
def test_band_step_fp32_keeps_the_spectrum(H, n, b, h):
    """Backward stable similarities: ||E||_2 <= 4 n eps32 ||A||_2."""
    import torch

    A = I.random_band(n, b, 13900 + n + b + h)
    A, got = reduce(H, A, b, h, torch.float32)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()


@pytest.mark.parametrize("n,b,h", [(700, 32, 16), (333, 32, 8), (450, 64, 16), (300, 24, 8), (200, 16, 4)])
def test_one_cta_and_several_give_the_same_bits(monkeypatch, n, b, h):
    import torch

    from paper_1604_03703_gb300 import api

    A = I.random_band(n, b, 14000 + n + b + h)
    outs = []
    for min_b in ("1", "1000"):
        monkeypatch.setenv("SEV_CHASE_X3_MIN_B", min_b)
        hd = api.Handle(0)
        outs.append(reduce(hd, A, b, h, torch.float32)[1])
        hd.close()
    np.testing.assert_array_equal(outs[0], outs[1])


@pytest.mark.parametrize("scale", [1e-150, 1e140])
def test_band_step_fp64_extreme_scales(H, orc, scale):
    import torch

    n, b, h = 150, 16, 4
    A = I.random_band(n, b, 14100)
    ref = orc.band_to_band(A, b, h)
    _, got = reduce(H, A * scale, b, h, torch.float64)
    np.testing.assert_allclose(np.tril(got) / scale, np.tril(ref), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)


@pytest.mark.parametrize("dtype_name,b", [("float32", 32), ("float32", 64), ("float64", 32)])
def test_wait_limit_runs_out_then_handle_still_works(H, dtype_name, b):
    import torch

    dt = getattr(torch, dtype_name)
    n, h = 1500, 16
    A = I.random_band(n, b, 14200)
    H.set_wait_limit(500)
    try:
        AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b).T)).to(dt).cuda()
        H.band_to_band(AB, b, h)
        assert H.get_error() == 3  # SEV_ERR_TIMEOUT
    finally:
        H.set_wait_limit(0)
    A, got = reduce(H, A, b, h, dt)
    lam = np.linalg.eigvalsh(A)
    eps = EPS32 if dtype_name == "float32" else EPS64
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * eps * np.abs(lam).max()
