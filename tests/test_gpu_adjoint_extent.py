"""The mixed adjoint of a compact set with one particle parked far away: the
position differences of close pairs do not depend on the extent of the system."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [0.0, 0.5])
@pytest.mark.parametrize("kind", ["plummer", "m4"])
@pytest.mark.parametrize("far", [1e2, 1e10, 1e14, 1e18, 1e20])
def test_core_with_a_parked_particle(far, kind, theta):
    """Against the FP64 adjoint on the same tree.  Float32 terms (6e-8, a few
    operations, r at the fifth power) with cancellations inside a pair: 1e-5 of
    the largest component, which belongs to the pair 0.01 apart (1 / r^3 = 1e6,
    the next pairs of the set at 0.05 and more).  The parked particle has no
    mass to speak of and no cotangent."""
    import torch
    from paper_2502_01496_gb300 import native
    rng = np.random.default_rng(17)
    x = rng.normal(size=(301, 3))
    x[1] = x[0] + 0.01 * np.array([0.6, -0.48, 0.64])
    x[-1] = far * np.array([0.3, 0.2, -0.9])
    m = np.full(301, 1.0 / 300)
    m[-1] = 1e-40
    b = rng.normal(size=(301, 3))
    b[-1] = 0.0
    h = np.full(301, 2e-3)
    cuda = lambda v: torch.tensor(v, device="cuda")
    res = []
    for precision in (native.FP64, native.MIXED):
        f = native.KdFmm(theta=theta, eps=1e-3, n_leaf=16, precision=precision,
                         soft_kind=native.SOFT_PLUMMER if kind == "plummer" else native.SOFT_M4)
        f.build(cuda(x), cuda(m), cuda(h) if kind == "m4" else None).accel()
        res.append([t.cpu().numpy() for t in f.vjp(cuda(b))])
    for want, got in zip(*res):
        assert np.isfinite(got).all()
        assert np.abs(got - want)[:-1].max() <= 1e-5 * np.abs(want)[:-1].max()
