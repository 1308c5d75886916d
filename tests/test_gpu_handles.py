"""Handles of different parameters living side by side in one process."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("other_leaf", [32, 1])
def test_a_handle_builds_again_after_another_with_other_leaves(other_leaf):
    """The subtree kernel's shared-memory limit is one value for the process:
    a second handle's leaf size must not take away what the first one needs."""
    import torch
    from paper_2502_01496_gb300 import native
    ps = wl.plummer(5000, 11)
    x = torch.tensor(ps.x, dtype=torch.float64, device="cuda")
    m = torch.tensor(ps.m, dtype=torch.float64, device="cuda")
    first = native.KdFmm(theta=0.5, eps=ps.eps, n_leaf=8, precision=native.FP64)
    first.build(x, m)
    a0, p0 = (t.clone() for t in first.accel())
    other = native.KdFmm(theta=0.5, eps=ps.eps, n_leaf=other_leaf, precision=native.FP64)
    other.build(x, m).accel()
    first.build(x, m)
    a1, p1 = first.accel()
    torch.cuda.synchronize()
    assert torch.equal(a0, a1) and torch.equal(p0, p1)
    assert np.isfinite(a1.cpu().numpy()).all()
