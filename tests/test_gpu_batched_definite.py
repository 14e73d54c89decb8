"""Definite matrices in the batched kernel: the bisection starts from the
Gershgorin interval itself, on one side of zero, as the oracle's does."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_definite_tridiagonal_is_bisected_bitwise(orc, sign):
    """FP32 tridiagonals pass through both reductions unchanged but for signs."""
    import torch

    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    dev, ref = [], []
    for k, n in enumerate([2, 3, 9, 33, 64, 129, 255]):
        r = I.rng(16500 + k)
        d = sign * (3.0 + r.random(n)).astype(np.float32).astype(np.float64)
        e = r.uniform(-1.0, 1.0, n - 1).astype(np.float32).astype(np.float64)
        dev.append(torch.from_numpy(np.diag(d) + np.diag(e, 1) + np.diag(e, -1)).float().cuda())
        ref.append(orc.bisect(d, e, 1e-9))
    got = [t.cpu().numpy() for t in h.eigvalsh_batched(dev, 8)]
    h.raise_device_error()
    h.close()
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)
