"""Kernels that wait within one launch, on several streams at once: band steps on
four CTAs a sweep, cooperative panels and bisections, whole solves.  Every wait
has a short limit; none runs out, and the results are those of each alone."""
import pytest

pytestmark = pytest.mark.gpu
LIMIT = 1_000_000_000  # ~0.5 s, some hundred times what any wait here takes


def test_band_steps_beside_cooperative_grids():
    import torch

    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(18400)

    def randn(*shape, dtype):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)

    def band(n, b, dtype):
        AB = randn(n, 2 * b, dtype=dtype)
        i, d = torch.arange(n, device="cuda")[:, None], torch.arange(2 * b, device="cuda")[None, :]
        AB[(d > b) | (i + d >= n)] = 0
        return AB

    def sym(n, dtype):
        A = randn(n, n, dtype=dtype)
        return A + A.T

    b1, b2, b3 = band(3000, 128, torch.float32), band(1500, 32, torch.float64), band(1200, 64, torch.float32)
    A1, A2 = sym(4600, torch.float32), sym(1300, torch.float64)
    d, e = randn(3000, dtype=torch.float64), randn(2999, dtype=torch.float64)
    work = [
        lambda h: [h.band_to_band(b1.clone(), 128, 32), h.band_to_band(b2.clone(), 32, 16), h.band_to_band(b3.clone(), 64, 16)],
        lambda h: [h.tridiag_bisect(d, e, 1e-12), h.full_to_band(A1.clone(), 64), h.tridiag_bisect(d, e, 1e-12)],
        lambda h: [h.eigvalsh(A2.clone()), h.tridiag_bisect(d, e, 1e-9)],
    ]
    handles = [api.Handle(0) for _ in work]
    ref = []
    for h, f in zip(handles, work):
        ref.append([t.clone() for t in f(h)])
        torch.cuda.synchronize()
        h.raise_device_error()
        h.set_wait_limit(LIMIT)
    streams = [torch.cuda.Stream() for _ in work]
    for _ in range(12):
        got = []
        for s, h, f in zip(streams, handles, work):
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                got.append(f(h))
        torch.cuda.synchronize()
        for h in handles:
            h.raise_device_error()
        for p, q in zip(got, ref):
            assert all(torch.equal(x, y) for x, y in zip(p, q))
    for h in handles:
        h.close()


def test_lanes_pass_after_pass():
    """A batch of large matrices run again and again with nothing waiting between."""
    import torch

    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(18500)
    h = api.Handle(0)
    h.set_wait_limit(LIMIT)
    sizes = [1281, 1538, 1792, 2049, 2306, 2560, 2817, 3074]
    A = []
    for n in sizes:
        a = torch.randn(n, n, generator=g, device="cuda")
        A.append(a + a.T)
    work = [a.clone() for a in A]
    outs = [torch.empty(n, dtype=torch.float64, device="cuda") for n in sizes]
    plan = h.batch_plan(work, outs)
    ref = None
    for _ in range(5):
        for _ in range(6):
            for w, a in zip(work, A):
                w.copy_(a)
            plan.run()
        h.raise_device_error()
        if ref is None:
            ref = [o.clone() for o in outs]
        assert all(torch.equal(o, r) for o, r in zip(outs, ref))
    h.close()
