"""One dual-walk handle rebuilt with other numbers of particles: its per-cell
buffers follow the tree it holds."""
import pytest

from paper_2502_01496_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_a_dual_handle_grows_with_its_particles(precision):
    """1, 300, 20011 and 700 particles through one handle give what a fresh handle
    gives for each, to the rounding that the order of the lists leaves (the lists
    are filled with atomics: per-cell sums of float64, or of float32 in mixed mode)."""
    import torch
    from paper_2502_01496_gb300 import native
    tol = 1e-12 if precision == native.FP64 else 2e-5
    kept = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16, precision=precision, walk=1)
    for n in (1, 300, 20011, 700):
        ps = W.plummer(n, W.seed_for(0, n))
        x = torch.tensor(ps.x, dtype=torch.float64, device="cuda")
        m = torch.tensor(ps.m, dtype=torch.float64, device="cuda")
        fresh = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16, precision=precision, walk=1)
        (a, p), (b, q) = kept.build(x, m).accel(), fresh.build(x, m).accel()
        torch.cuda.synchronize()
        assert (a - b).norm(dim=1).max() <= tol * b.norm(dim=1).max()
        assert (p - q).abs().max() <= tol * q.abs().max()
        assert torch.isfinite(a).all() and torch.isfinite(p).all()
