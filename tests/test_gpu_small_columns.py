"""Reflectors of columns far from order one, in every path that forms them from
unscaled squares: couplings whose squares underflow beside entries of order one
(a reflector that is not orthogonal there spoils the large entries), and whole
matrices at such scales (where dropping the column loses it)."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = {"float64": 2.0**-52, "float32": 2.0**-23}
# norms whose squares are normal, subnormal, zero
TINY = {"float64": [1e-140, 1e-150, 1e-153, 1e-155, 1e-157, 1e-160, 1e-170, 1e-300, 1e-310],
        "float32": [1e-17, 1e-19, 1e-20, 1e-21, 1e-22, 1e-24, 1e-30, 1e-40]}
SCALES = {"float64": [1e-157, 1e-170, 1e-250, 1e160, 1e250],
          "float32": [1e-20, 1e-22, 1e-25, 1e-30, 1e20, 1e25, 1e30]}


@pytest.fixture(scope="module")
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def cases(table):
    return [(dt, v) for dt in table for v in table[dt]]


def couple(A, cuts, c):
    """A with its entries across every cut (rows >= k, columns < k) scaled by c."""
    A = A.copy()
    for k in cuts:
        A[k:, :k] *= c
        A[:k, k:] *= c
    return A


def to_1(H, A, b, dt):
    """b -> 1 on the GPU: the band it got and the tridiagonal, in float64."""
    import torch

    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b).T)).to(getattr(torch, dt)).cuda()
    A = I.band_to_dense(AB.double().cpu().numpy().T)
    H.band_to_band(AB, b, 1)
    H.raise_device_error()
    return A, I.band_to_dense(AB.double().cpu().numpy().T)


def bound(n, dt, A):
    """n reductions by orthogonal similarities, each backward stable."""
    return 4 * n * EPS[dt] * np.linalg.norm(A)


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("dt,c", cases(TINY))
def test_band_to_1_with_tiny_couplings(H, dt, c, b):
    n = 70
    A = couple(I.random_band(n, b, 17000 + b), [1, 2, b + 2, 40], c)
    A, T = to_1(H, A, b, dt)
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(T) - lam).max() <= bound(n, dt, A)


def test_band_to_1_two_vector(H):
    """The smallest case, its sum of squares subnormal: the 2 x 2 block that is
    left over keeps its eigenvalues."""
    A = np.array([[1.0, 6e-156, 8e-156], [6e-156, 1.0, 0.5], [8e-156, 0.5, -2.0]])
    A, T = to_1(H, A, 2, "float64")
    np.testing.assert_allclose(np.linalg.eigvalsh(T), np.linalg.eigvalsh(A), atol=bound(3, "float64", A), rtol=0)


@pytest.mark.parametrize("b", [2, 8, 16])
@pytest.mark.parametrize("dt,scale", cases(SCALES))
def test_band_to_1_at_extreme_scales(H, dt, scale, b):
    n = 70
    A, T = to_1(H, I.random_band(n, b, 17100 + b) * scale, b, dt)
    A, T = A / scale, T / scale
    lam = np.linalg.eigvalsh(A)
    assert np.abs(np.linalg.eigvalsh(T) - lam).max() <= bound(n, dt, A)


@pytest.mark.parametrize("dt,c", cases(TINY))
def test_eigvalsh_and_batch_with_tiny_couplings(H, dt, c):
    """The whole solve, and the batched kernel (whose panels are its own)."""
    import torch

    n = 90
    for cuts in ([1], [3], [8], [16, 40]):
        A = couple(I.semicircle(n, 17200), cuts, c)
        t = torch.from_numpy(A).to(getattr(torch, dt))
        lam = np.linalg.eigvalsh(t.double().numpy())
        one = H.eigvalsh(t.cuda(), 8).cpu().numpy()
        batch = [H.eigvalsh_batched([t.cuda()], b)[0].cpu().numpy() for b in (4, 8, 16)]
        H.raise_device_error()
        for got in [one] + batch:
            assert np.abs(got - lam).max() <= bound(n, dt, A), cuts


@pytest.mark.parametrize("dt,scale", cases(SCALES))
def test_eigvalsh_and_batch_at_extreme_scales(H, dt, scale):
    import torch

    n = 90
    A = I.semicircle(n, 17300)
    t = torch.from_numpy(A * scale).to(getattr(torch, dt))
    lam = np.linalg.eigvalsh(t.double().numpy() / scale)
    one = H.eigvalsh(t.cuda(), 8).cpu().numpy()
    batch = [H.eigvalsh_batched([t.cuda()], b)[0].cpu().numpy() for b in (4, 8, 16)]
    H.raise_device_error()
    for got in [one] + batch:
        assert np.abs(got / scale - lam).max() <= bound(n, dt, A)


@pytest.mark.parametrize("dt,c", cases(TINY))
def test_tree_panels_with_tiny_couplings(monkeypatch, dt, c):
    """The tree QR's register leaves (b = 16, 12) and shared-memory ones (b = 5);
    a column whose leading entry is zero."""
    import torch

    from paper_1604_03703_gb300 import api

    monkeypatch.setenv("SEV_LEAF_ROWS", "64")
    h = api.Handle(0)
    n = 200
    for b in (16, 12, 5):
        for k in (1, b, b + 1):
            A = couple(I.semicircle(n, 17400 + b), [k], c)
            A[b, 0] = A[0, b] = 0.0
            t = torch.from_numpy(A).to(getattr(torch, dt))
            A = t.double().numpy()
            band = I.band_to_dense(h.full_to_band(t.cuda(), b).double().cpu().numpy().T)
            h.raise_device_error()
            assert np.all(np.isfinite(band)), (b, k)
            assert np.abs(np.linalg.eigvalsh(band) - np.linalg.eigvalsh(A)).max() <= bound(n, dt, A), (b, k)
    h.close()


# a matrix far from order one whose columns are far smaller still: x^T a of a block
# that is not held scaled underflows before 1 / (alpha - beta) brings it back
BOTH = [("float64", 1e-170, 1e-130), ("float64", 1e-190, 1e-120), ("float64", 1e-190, 1e-135), ("float64", 1e-230, 1e-75),
        ("float64", 1e200, 1e-135), ("float32", 1e-22, 1e-14), ("float32", 1e-26, 1e-12), ("float32", 1e-30, 1e-7), ("float32", 1e25, 1e-14)]


@pytest.mark.parametrize("b,h", [(8, 2), (32, 16), (64, 16), (64, 32), (96, 32), (128, 16)])
@pytest.mark.parametrize("dt,scale,c", BOTH)
def test_band_steps_with_both(H, dt, scale, c, b, h):
    import torch

    n = 3 * b + 20
    A = couple(I.random_band(n, b, 17500 + b + h), [1, h, h + 1, b, b + 3, 2 * b + 1], c) * scale
    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b).T)).to(getattr(torch, dt)).cuda()
    A = I.band_to_dense(AB.double().cpu().numpy().T) / scale
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    G = I.band_to_dense(AB.double().cpu().numpy().T) / scale
    assert np.abs(np.linalg.eigvalsh(G) - np.linalg.eigvalsh(A)).max() <= bound(n, dt, A)


@pytest.mark.parametrize("n,b", [(90, 8), (300, 32), (300, 64), (1300, 16), (2300, 64)])
@pytest.mark.parametrize("dt,scale,c", BOTH)
def test_panels_with_both(H, dt, scale, c, n, b):
    """One cluster and the whole GPU (FP64 over 1024 rows)."""
    import torch

    if n == 2300 and dt == "float64":
        pytest.skip("an order is enough")
    A = couple(I.semicircle(n, 17600 + n), [1, b, b + 1, 2 * b + 5, n - 3], c) * scale
    t = torch.from_numpy(A).to(getattr(torch, dt))
    A = t.double().numpy() / scale
    G = I.band_to_dense(H.full_to_band(t.cuda(), b).double().cpu().numpy().T) / scale
    H.raise_device_error()
    assert np.abs(np.linalg.eigvalsh(G) - np.linalg.eigvalsh(A)).max() <= bound(n, dt, A)


@pytest.mark.parametrize("n,b,h", [(816, 110, 22), (700, 64, 16), (600, 32, 16), (800, 128, 16), (500, 16, 4), (900, 48, 24)])
@pytest.mark.parametrize("k", [-540, -600, -634, -680])
def test_sparse_bands_far_below_one(H, k, n, b, h):
    """Few entries: the columns left by earlier sweeps are rounding errors of rounding
    errors, 2^-53, 2^-106, ... of their block, down to the end of the range."""
    import torch

    for seed in range(4):
        r = I.rng(19000 + 10 * b + seed)
        A = np.where(r.random((n, n)) < 0.03, r.standard_normal((n, n)), 0.0)
        A = np.tril(A) + np.tril(A, -1).T
        i, j = np.indices(A.shape)
        A[np.abs(i - j) > b] = 0.0
        AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A * 2.0**k, 2 * b).T)).cuda()
        H.band_to_band(AB, b, h)
        H.raise_device_error()
        G = I.band_to_dense(AB.cpu().numpy().T) / 2.0**k
        assert np.abs(np.linalg.eigvalsh(G) - np.linalg.eigvalsh(A)).max() <= bound(n, "float64", A), seed


@pytest.mark.parametrize("n,b", [(300, 32), (816, 64), (1300, 16)])
@pytest.mark.parametrize("k", [-540, -600, -634, -680])
def test_sparse_matrices_far_below_one(H, k, n, b):
    import torch

    for seed in range(3):
        r = I.rng(19100 + 10 * b + seed)
        A = np.where(r.random((n, n)) < 2.0 / n, r.standard_normal((n, n)), 0.0)
        A = np.tril(A) + np.tril(A, -1).T
        G = I.band_to_dense(H.full_to_band(torch.from_numpy(A * 2.0**k).cuda(), b).cpu().numpy().T) / 2.0**k
        H.raise_device_error()
        assert np.abs(np.linalg.eigvalsh(G) - np.linalg.eigvalsh(A)).max() <= bound(n, "float64", A), seed
