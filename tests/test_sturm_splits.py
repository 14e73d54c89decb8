"""Tridiagonals that split behind a block singular at a midpoint of the bisection
(zero is one as soon as the Gershgorin interval is symmetric): from there on all
leading principal minors vanish.  diag(0, 1, -1) is the smallest."""
import ctypes

import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I


def cases():
    out = [([0.0, 1.0, -1.0], [0.0, 0.0]), ([0.0, 0.0, 0.0, 1.0, -1.0], [1.0, 1.0, 0.0, 0.0]), ([0.0] * 4 + [1.0], [1.0, 0.0, 1.0, 0.0]),
           ([0.0, 0.0, 0.0], [0.0, 1.0]), ([0.5, -0.5, 0.0, 0.0, 1.0, -1.0], [0.5, 0.0, 0.0, 0.0, 0.0]), ([1.0, 0.0, -1.0], [0.0, 0.0])]
    r = I.rng(18800)
    for n in (9, 10, 17, 40, 300, 2049):
        d = r.choice([0.0, 0.0, 1.0, -1.0, 0.5], n)
        e = r.choice([0.0, 0.0, 1.0, 0.25], n - 1)
        d[-2:], e[-1] = (2.0, -2.0), 0.0  # the symmetric interval
        e[-2] = 0.0
        out.append((d, e))
        # couplings that are not zero but vanish in the products
        out.append((d, np.where(e == 0.0, 1e-140, e)))
        out.append((d, np.where(e == 0.0, 1e-170, e)))
    return [(np.array(d), np.array(e)) for d, e in out]


def check(got, d, e, rtol):
    lam = np.linalg.eigvalsh(np.diag(d) + np.diag(e, 1) + np.diag(e, -1))
    norm = np.abs(lam).max()
    assert np.abs(got - lam).max() <= (2 * rtol + 50 * 2.0**-52 * len(d) ** 0.5) * norm


@pytest.mark.parametrize("k", range(len(cases())))
def test_oracle(orc, k):
    d, e = cases()[k]
    check(orc.bisect(d, e, 1e-13), d, e, 1e-13)


@pytest.mark.gpu
def test_bisection_paths(orc):
    import torch

    from paper_1604_03703_gb300 import _lib, api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h, lib = api.Handle(0), _lib.load()
    for d, e in cases():
        dt, et = torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda()
        got = h.tridiag_bisect(dt, et, 1e-13)
        h.raise_device_error()
        check(got.cpu().numpy(), d, e, 1e-13)
        np.testing.assert_array_equal(got.cpu().numpy(), orc.bisect(d, e, 1e-13))
        out = torch.empty_like(dt)
        assert lib.sev_tridiag_bisect_static(len(d), ctypes.c_void_p(dt.data_ptr()), ctypes.c_void_p(et.data_ptr()), 1e-13,
                                             ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert torch.equal(out, got)
    h.close()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
def test_sparse_matrices(dtype_name):
    """Whole solves and batches: isolated rows, hollow and diagonal matrices."""
    import torch

    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    dt, eps, rtol = (torch.float64, 2.0**-52, 1e-14) if dtype_name == "float64" else (torch.float32, 2.0**-23, 1e-9)
    mats = [np.diag([0.0, 1.0, -1.0]), np.diag([1.0, 0.0, -1.0, 0.0, 0.5])]
    for k, n in enumerate([2, 3, 4, 5, 8, 13, 21, 40, 120] * 4):
        r = I.rng(18900 + k)
        A = np.where(r.random((n, n)) < 0.15, r.choice([1.0, -1.0, 0.5], (n, n)), 0.0)
        A = np.tril(A, -1) + np.tril(A, -1).T + (np.diag(r.choice([0.0, 1.0, -1.0], n)) if k % 2 else 0.0)
        mats.append(A)
    dev = [torch.from_numpy(A).to(dt).cuda() for A in mats]
    got = {b: h.eigvalsh_batched([t.clone() for t in dev], b) for b in (4, 8, 16)}
    for i, A in enumerate(mats):
        n = A.shape[0]
        lam = np.linalg.eigvalsh(A)
        bound = (8 * n * eps + 2 * rtol) * max(np.linalg.norm(A), 1.0)
        for g in [h.eigvalsh(dev[i].clone(), 8), h.eigvalsh(dev[i].clone())] + [got[b][i] for b in got]:
            assert np.abs(g.cpu().numpy() - lam).max() <= bound, (i, n)
    h.raise_device_error()
    h.close()
