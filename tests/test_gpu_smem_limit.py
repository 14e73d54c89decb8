"""The limit of a kernel's dynamic shared memory belongs to the process, not to
the call that sets it: a call with a smaller need in between takes nothing away."""
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


@pytest.mark.parametrize("dtype_name,b", [("float32", 16), ("float64", 8)])
def test_large_plan_runs_after_a_small_one_was_made(H, dtype_name, b):
    import torch

    g = torch.Generator(device="cuda")
    g.manual_seed(16400)
    plans = []
    for n in (500, 60):
        A = torch.randn(n, n, generator=g, device="cuda", dtype=getattr(torch, dtype_name))
        A = A + A.T
        out = torch.zeros(n, dtype=torch.float64, device="cuda")
        work = A.clone()
        plans.append((A, work, out, H.batch_plan([work], [out], b)))
    for A, work, out, plan in plans + plans[:1]:
        out.zero_()
        work.copy_(A)
        plan.run()
        H.raise_device_error()
        lam = torch.linalg.eigvalsh(A.double().cpu())
        eps = 2.0**-23 if dtype_name == "float32" else 2.0**-52
        assert (out.cpu() - lam).abs().max() <= 4 * A.shape[0] * eps * A.double().norm().cpu()


def test_large_plan_runs_after_the_batch_autotuner(H):
    import torch

    n = 500
    A = torch.randn(n, n, device="cuda")
    A = A + A.T
    work = A.clone()
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    plan = H.batch_plan([work], [out], 16)
    H.batch_autotune([50, 60, 70], 1)
    plan.run()
    H.raise_device_error()
    lam = torch.linalg.eigvalsh(A.double().cpu())
    assert (out.cpu() - lam).abs().max() <= 4 * n * 2.0**-23 * A.double().norm().cpu()
