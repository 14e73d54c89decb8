"""The cooperative panel factorisation where it can go wrong: edges of the rows
per CTA, one to many CTAs, widths that are no multiple of a warp, fewer rows
than columns, zero and tiny columns, entries near the ends of the FP64 range."""
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


def f2b(H, A, b, dtype):
    import torch

    AB = H.full_to_band(torch.from_numpy(np.ascontiguousarray(A)).to(dtype).cuda(), b)
    H.raise_device_error()
    return I.band_to_dense(AB.double().cpu().numpy().T)


# b + 1 .. b + 64 .. : the first panel has 1, 63, 64, 65, 128 rows etc.; widths off the warp grid
@pytest.mark.parametrize("n,b", [(9, 7), (33, 31), (40, 33), (95, 32), (96, 32), (97, 32), (129, 64), (128, 64),
                                 (193, 64), (170, 17), (300, 48), (200, 1), (150, 5), (600, 63)])
def test_panel_fp64_vs_oracle(H, orc, n, b):
    import torch

    A = I.semicircle(n, 13200 + n + b)
    ref = orc.full_to_band(A, b)
    got = f2b(H, A, b, torch.float64)
    np.testing.assert_allclose(np.tril(got), np.tril(ref), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)


@pytest.mark.parametrize("n,b", [(257, 128), (400, 127), (513, 100), (300, 33), (1200, 96), (2300, 128), (4300, 64), (90, 8),
                                 (70, 3)])
def test_panel_fp32_keeps_the_spectrum(H, n, b):
    """Backward stable similarities: ||E||_2 <= 4 n eps32 ||A||_2 (the bound of
    the other FP32 full-to-band test)."""
    import torch

    A = I.semicircle(n, 13300 + n + b).astype(np.float32).astype(np.float64)
    got = f2b(H, A, b, torch.float32)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > b] == 0.0)


@pytest.mark.parametrize("scale", [1e-200, 1e-150, 1e140])
def test_panel_fp64_extreme_scales(H, orc, scale):
    """Squares of the entries over- or underflow; the reduction is scale-free."""
    import torch

    n, b = 200, 16
    A = I.semicircle(n, 13400)
    ref = orc.full_to_band(A, b)
    got = f2b(H, A * scale, b, torch.float64)
    np.testing.assert_allclose(np.tril(got) / scale, np.tril(ref), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)


@pytest.mark.parametrize("dtype_name", ["float64", "float32"])
@pytest.mark.parametrize("kind", ["zero", "rank1", "block", "graded"])
def test_panel_degenerate_columns(H, kind, dtype_name):
    """Zero columns (tau = 0), columns of rounding noise, columns 1e-200 times
    smaller than their neighbours: the spectrum stays within 4 n eps ||A||_2."""
    import torch

    n, b = 260, 32
    r = I.rng(13500)
    if kind == "zero":
        A = np.zeros((n, n))
    elif kind == "rank1":
        v = r.standard_normal(n)
        A = np.outer(v, v) / n
    elif kind == "block":
        A = np.zeros((n, n))
        A[:100, :100] = I.semicircle(100, 13501)
        A[200:, 200:] = I.semicircle(60, 13502)
    else:
        g = 10.0 ** np.linspace(0, -200 if dtype_name == "float64" else -12, n)
        A = I.semicircle(n, 13503) * np.sqrt(np.outer(g, g))
    dt = getattr(torch, dtype_name)
    A = torch.from_numpy(A).to(dt).double().numpy()
    got = f2b(H, A, b, dt)
    lam = np.linalg.eigvalsh(A)
    eps = EPS64 if dtype_name == "float64" else EPS32
    assert np.all(np.isfinite(got))
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * eps * max(np.abs(lam).max(), 1e-300)


def test_panel_wait_limit_runs_out_then_handle_still_solves(H, orc):
    """A limit of a few cycles ends the CTAs' first wait for one another; the
    error is latched, every CTA leaves, and the handle works again."""
    import torch

    n, b = 700, 32
    A = I.semicircle(n, 13600)
    H.set_wait_limit(1)
    try:
        H.full_to_band(torch.from_numpy(A).cuda(), b)
        assert H.get_error() == 3  # SEV_ERR_TIMEOUT
    finally:
        H.set_wait_limit(0)
    got = f2b(H, A, b, torch.float64)
    np.testing.assert_allclose(np.tril(got), np.tril(orc.full_to_band(A, b)), atol=20 * n * EPS64 * np.linalg.norm(A), rtol=0)
