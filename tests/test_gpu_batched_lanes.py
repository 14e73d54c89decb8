"""Large matrices of a batch run side by side on streams of the handle's own:
the results are those of one call per matrix, bit for bit, and later work on
the caller's stream waits for them."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
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


@pytest.mark.parametrize("dtype_name,sizes", [("float32", [1025, 1100, 1531, 1200, 1040, 64, 1301]),
                                              ("float32", [4100, 1100, 1200]), ("float64", [1030, 1100]),
                                              ("float32", [1400])])
def test_side_by_side_is_bitwise(H, dtype_name, sizes):
    import torch

    A = matrices(torch, sizes, getattr(torch, dtype_name), 16100)
    ref = [H.eigvalsh(a.clone()).clone() for a, n in zip(A, sizes) if n > 1024]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        work = [a.clone() for a in A]
        outs = [torch.empty(n, dtype=torch.float64, device="cuda") for n in sizes]
        plan = H.batch_plan(work, outs)
        for _ in range(3):  # the copies wait for the previous run, the run for the copies
            for w, a in zip(work, A):
                w.copy_(a)
            plan.run()
            got = [o.clone() for o, n in zip(outs, sizes) if n > 1024]
            for o in outs:
                o.zero_()
            for a, b in zip(got, ref):
                assert torch.equal(a, b)
    H.raise_device_error()
