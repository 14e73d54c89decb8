"""Panels of different widths on clusters of the same size, on one handle: what it
has learnt for one kernel is not taken for another."""
import numpy as np
import pytest

from paper_1604_03703_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype_name,shapes", [("float32", [(4095, 32), (2047, 128), (4095, 64), (2047, 96)]),
                                               ("float64", [(1023, 8), (1023, 64)])])
def test_widths_share_a_handle(dtype_name, shapes):
    """Full clusters of 16 CTAs first: the bits are those of a handle of its own."""
    import torch

    from paper_1604_03703_gb300 import api
    from paper_1604_03703_gb300 import build as B

    B.build()
    h = api.Handle(0)
    for n, b in shapes:
        A = torch.from_numpy(I.semicircle(n, 17800 + b)).to(getattr(torch, dtype_name)).cuda()
        got = h.full_to_band(A.clone(), b)
        h.raise_device_error()
        own = api.Handle(0)
        ref = own.full_to_band(A.clone(), b)
        own.raise_device_error()
        own.close()
        assert torch.equal(got, ref)
        assert bool(torch.isfinite(got).all())
    h.close()
