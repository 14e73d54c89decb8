"""A band reduction needs little workspace; the exchange buffers of the faster
kernel are a wish: a caller's workspace without room for them is enough, and the
handle's own is not replaced for them."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = {"float32": 2.0**-23, "float64": 2.0**-52}


@pytest.fixture()
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def band(n, b, dtype_name):
    import torch

    A = I.random_band(n, b, 18600 + n + b)
    AB = torch.from_numpy(np.ascontiguousarray(I.dense_to_band(A, 2 * b).T)).to(getattr(torch, dtype_name)).cuda()
    return AB, I.band_to_dense(AB.double().cpu().numpy().T)


def check(AB, A, h, dtype_name):
    got = I.band_to_dense(AB.double().cpu().numpy().T)
    i, j = np.indices(got.shape)
    assert np.all(got[np.abs(i - j) > h] == 0.0)
    lam = np.linalg.eigvalsh(A)
    n = A.shape[0]
    assert np.abs(np.linalg.eigvalsh(got) - lam).max() <= 4 * n * EPS[dtype_name] * np.abs(lam).max()


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
@pytest.mark.parametrize("n,b,h", [(500, 64, 16), (300, 32, 16), (260, 96, 8), (200, 6, 3)])
def test_small_workspace_of_the_caller(H, dtype_name, n, b, h):
    import torch

    AB, A = band(n, b, dtype_name)
    ws = torch.empty(16384, dtype=torch.uint8, device="cuda")  # a progress counter per sweep and one more
    H.set_workspace(ws)
    try:
        H.band_to_band(AB, b, h)
        H.raise_device_error()
    finally:
        H.set_workspace(None)
    check(AB, A, h, dtype_name)
    AB, A = band(n, b, dtype_name)
    H.band_to_band(AB, b, h)
    H.raise_device_error()
    check(AB, A, h, dtype_name)


def test_workspace_too_small_for_the_chase_is_refused(H):
    import torch

    AB, _ = band(500, 64, "float32")
    H.set_workspace(torch.empty(256, dtype=torch.uint8, device="cuda"))
    try:
        with pytest.raises(Exception, match="WORKSPACE"):
            H.band_to_band(AB, 64, 16)
    finally:
        H.set_workspace(None)


def test_graph_outlives_a_band_reduction(H):
    """The graph of a small solve, replayed after a band reduction with larger
    exchange buffers than the workspace it refers to."""
    import torch

    n = 300
    A = torch.from_numpy(I.semicircle(n, 18700)).float().cuda()
    ref = H.eigvalsh(A.clone()).clone()
    H.raise_device_error()
    work, out = A.clone(), torch.zeros(n, dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        H.eigvalsh(work, 0, out)
    own = H.workspace_query(n, 0, 1)
    n2, b = 6000, 128
    slots = min(min((n2 - 2 - 8) // b // 2 + 4, 160), (n2 - 2) // 8)
    assert slots * 4 * 8 * (2 * 132 * 8 + 12 * 128) > own  # the exchange buffers of 128 -> 8 would have replaced it
    AB, _ = band(n2, b, "float32")
    H.band_to_band(AB, b, 8)
    H.raise_device_error()
    work.copy_(A)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_captured_with_the_workspace_at_hand(H):
    import torch

    AB0, A = band(400, 64, "float64")
    H.tridiag_bisect(torch.ones(400, dtype=torch.float64, device="cuda"), torch.ones(399, dtype=torch.float64, device="cuda"))
    H.raise_device_error()
    AB = AB0.clone()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        H.band_to_band(AB, 64, 16)
    for _ in range(2):
        AB.copy_(AB0)
        g.replay()
        torch.cuda.synchronize()
        check(AB, A, 16, "float64")
    H.raise_device_error()
