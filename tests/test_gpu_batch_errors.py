"""A non-finite matrix spoils its own result only: what runs beside it, behind it
in the batch or behind it on the handle gives the bits it gives alone, and the
handle still reports the error."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture()
def H():
    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    yield h
    h.close()


def matrices(torch, sizes, dt, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = []
    for n in sizes:
        L = torch.tril(torch.randn(n, n, generator=g, device="cuda", dtype=dt))
        out.append(L + torch.tril(L, -1).T)
    return out


# side by side on the handle's lanes, and one on the handle's own stream
@pytest.mark.parametrize("dtype_name,sizes,bad", [("float32", [1301, 1200, 1531, 1100, 1040, 1025, 1400, 1240, 1150], 2),
                                                  ("float32", [1301, 1200, 1100, 1040], 3),
                                                  ("float64", [1030, 1100, 1060], 0),
                                                  ("float32", [4200, 1200], 0),
                                                  # in the batched launch
                                                  ("float32", [64, 100, 1200, 33], 1), ("float64", [64, 100, 33], 2)])
def test_nan_in_one_matrix_of_a_batch(H, dtype_name, sizes, bad):
    import torch

    A = matrices(torch, sizes, getattr(torch, dtype_name), 16200)
    outs = [torch.zeros(n, dtype=torch.float64, device="cuda") for n in sizes]
    work = [a.clone() for a in A]
    plan = H.batch_plan(work, outs)

    def run(spoil):
        for i, (w, a) in enumerate(zip(work, A)):
            w.copy_(a)
            if spoil and i == bad:
                w[sizes[i] // 2, 3] = w[3, sizes[i] // 2] = float("nan")
        plan.run()
        return [o.clone() for o in outs]

    ref = run(False)
    assert H.get_error() == 0
    for _ in range(3):
        got = run(True)
        assert H.get_error() == 1  # SEV_ERR_NONFINITE
        for i, (g, r) in enumerate(zip(got, ref)):
            if i == bad:
                assert bool(torch.isnan(g).all())
            else:
                assert torch.equal(g, r), sizes[i]


@pytest.mark.parametrize("b", [4, 8, 16])
@pytest.mark.parametrize("n,i,j,value", [(1, 0, 0, "nan"), (2, 0, 0, "inf"), (2, 1, 0, "nan"), (5, 4, 4, "-inf"),
                                         (40, 39, 0, "nan"), (200, 199, 199, "nan"), (200, 0, 0, "inf"), (200, 101, 100, "nan")])
def test_nonfinite_entry_of_a_small_matrix(H, n, i, j, value, b):
    """Latched, and no eigenvalue is finite (n = 1: the entry itself)."""
    import torch

    (A,) = matrices(torch, [n], torch.float32, 16260)
    A[i, j] = A[j, i] = float(value)
    got = H.eigvalsh_batched([A], b)[0]
    assert H.get_error() == 1  # SEV_ERR_NONFINITE
    assert not bool(torch.isfinite(got).any())


def test_overflow_inside_the_reduction_is_not_silent(H):
    """Finite entries whose products overflow FP32."""
    import torch

    n = 100
    A = torch.full((n, n), 3e38, device="cuda")
    got = H.eigvalsh_batched([A], 8)[0]
    assert H.get_error() == 1  # SEV_ERR_NONFINITE
    assert bool(torch.isnan(got).all())


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
def test_nothing_finite_from_a_solve_whose_waits_ran_out(H, dtype_name):
    """Until the error has been read; then the handle solves as before."""
    import torch

    n = 1300
    (A,) = matrices(torch, [n], getattr(torch, dtype_name), 16250)
    ref = H.eigvalsh(A.clone())
    assert H.get_error() == 0
    H.set_wait_limit(1)
    try:
        first = H.eigvalsh(A.clone())
    finally:
        H.set_wait_limit(0)
    second = H.eigvalsh(A.clone())
    assert H.get_error() == 3  # SEV_ERR_TIMEOUT
    assert bool(torch.isnan(first).all()) and bool(torch.isnan(second).all())
    assert torch.equal(H.eigvalsh(A.clone()), ref)
    assert H.get_error() == 0


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
def test_call_after_a_nan_whose_error_was_not_read(H, dtype_name):
    import torch

    n = 1300
    A, B = matrices(torch, [n, n], getattr(torch, dtype_name), 16300)
    ref = H.eigvalsh(B.clone())
    assert H.get_error() == 0
    A[700, 11] = A[11, 700] = float("nan")
    bad = H.eigvalsh(A)
    got = H.eigvalsh(B.clone())
    assert H.get_error() == 1  # SEV_ERR_NONFINITE
    assert bool(torch.isnan(bad).all())
    assert torch.equal(got, ref)
