"""FP32 matrices without 16-byte aligned columns are reduced in an aligned copy.
The buffer for it is no part of what a captured graph refers to, is not
allocated under capture, and a batch plan has it before it runs."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)


@pytest.fixture()
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def strided(A, ld):
    import torch

    n = A.shape[0]
    t = torch.zeros(n * ld, dtype=torch.float32, device="cuda").view(n, ld)[:, :n]
    t.copy_(torch.from_numpy(A).float())
    return t


def capture(H, t, b0, out):
    import torch

    work = t.clone() if t.is_contiguous() else torch.empty_strided(t.shape, t.stride(), dtype=t.dtype, device=t.device)
    g = torch.cuda.CUDAGraph()
    work.copy_(t)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        H.eigvalsh(work, b0, out)
    return g, work


def test_unaligned_call_is_captured_after_an_aligned_one(H):
    import torch

    n, b0 = 1101, 64
    A = I.semicircle(n, 17500).astype(np.float32).astype(np.float64)
    lam = np.linalg.eigvalsh(A)
    H.eigvalsh(strided(A, 1104), b0)
    H.raise_device_error()
    t, out = strided(A, n), torch.zeros(n, dtype=torch.float64, device="cuda")
    g, work = capture(H, t, b0, out)
    for _ in range(2):
        out.zero_()
        work.copy_(t)
        g.replay()
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - lam).max() <= 4 * n * EPS32 * np.abs(lam).max()
    H.raise_device_error()


def test_graph_outlives_an_unaligned_call(H):
    """The graph of an aligned solve, replayed after an unaligned call of the same
    order: the workspace it refers to is still the handle's."""
    import torch

    n, b0 = 1101, 64
    A = I.semicircle(n, 17600).astype(np.float32).astype(np.float64)
    t = strided(A, 1104)
    ref = H.eigvalsh(strided(A, 1104), b0).clone()
    H.raise_device_error()
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    g, work = capture(H, t, b0, out)
    free = torch.cuda.mem_get_info()[0]
    H.eigvalsh(strided(A, n), b0)
    H.raise_device_error()
    assert free - torch.cuda.mem_get_info()[0] < 16 << 20  # the copy (5 MB), not a second workspace
    work.copy_(t)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_plan_of_unaligned_matrices_runs_without_allocating(H):
    import torch

    sizes = [1101, 1203, 1305, 2051]
    mats = [torch.from_numpy(I.semicircle(n, 17700 + n)).float().cuda() for n in sizes]
    outs = [torch.zeros(n, dtype=torch.float64, device="cuda") for n in sizes]
    plan = H.batch_plan(mats, outs)
    lam = [np.linalg.eigvalsh(m.double().cpu().numpy()) for m in mats]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan.run()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    H.raise_device_error()
    for n, o, r in zip(sizes, outs, lam):
        assert np.abs(o.cpu().numpy() - r).max() <= 4 * n * EPS32 * np.abs(r).max()
