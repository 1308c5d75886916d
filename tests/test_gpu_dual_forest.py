"""The dual walk over forests on both sides of its limit of two systems (one
block for the first levels of the pair recursion and of the downward pass)."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_sys", [1, 2, 3, 4, 5, 300])
def test_forest_against_the_oracle(oracle, n_sys, precision):
    """Systems of 1 to 400 particles and one of 6000, theta from 0.3 to 0.8, against
    the oracle's dual walk of each; the precisions' bounds, against the system's
    largest value (a particle's own may cancel)."""
    import torch
    from paper_2502_01496_gb300 import native
    rng = np.random.default_rng(n_sys)
    sizes = np.append(6000, rng.integers(1, 400, n_sys - 1))
    theta = rng.uniform(0.3, 0.8, n_sys)
    systems = [W.plummer(int(n), 200 + k) for k, n in enumerate(sizes)]
    off = np.append(0, np.cumsum(sizes))
    cuda = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")
    f = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16, precision=precision, walk=1)
    f.build_forest(cuda(np.concatenate([p.x for p in systems])), cuda(np.concatenate([p.m for p in systems])),
                   None, off, theta=theta)
    a, phi = (t.cpu().numpy() for t in f.accel())
    tol = 1e-12 if precision == 0 else 2e-5
    for p, th, i, j in zip(systems, theta, off, off[1:]):
        T = oracle.Tree(p.x, p.m, None, theta=th, n_leaf=16, soft_kind=0, eps=0.01)
        wa, wphi = T.eval_dual()
        assert np.abs(a[i:j] - wa).max() <= tol * np.abs(wa).max(), (i, j)
        assert np.abs(phi[i:j] - wphi).max() <= tol * np.abs(wphi).max(), (i, j)
