"""Float64 near-field kernels with everything near (theta = 0): leaves of 1 to 32
particles fill a staged chunk in every way (one leaf of a chunk to 32), and
supports that hold none, some or all of the pairs fill the queue of inside pairs
never, partly or beyond its 512 marks."""
import numpy as np
import pytest

from test_gpu_adjoint_lists import _direct

pytestmark = pytest.mark.gpu


def _set(n, scale, seed=3):
    g = np.random.default_rng(seed)
    return g.normal(size=(n, 3)), g.uniform(0.5, 1.5, n) / n, scale * g.uniform(0.5, 1.5, n)


# float64 sums of at most 700 terms: 1e-12 of the largest component
@pytest.mark.parametrize("scale", [1e-3, 0.3, 50.0])
@pytest.mark.parametrize("n,n_leaf", [(2, 1), (33, 1), (700, 1), (700, 2), (650, 7), (512, 16), (700, 31), (700, 32)])
def test_near_pairs_of_the_direct_sum(oracle, n, n_leaf, scale):
    import torch
    from paper_2502_01496_gb300 import native
    x, m, h = _set(n, scale)
    f = native.KdFmm(theta=0.0, eps=0.01, n_leaf=n_leaf, soft_kind=native.SOFT_M4, precision=native.FP64)
    f.build(*(torch.tensor(v, device="cuda") for v in (x, m, h)))
    a, phi = (t.cpu().numpy() for t in f.accel())
    wa, wphi = oracle.direct(x, m, h, soft_kind=native.SOFT_M4)
    assert np.abs(a - wa).max() < 1e-12 * np.abs(wa).max()
    assert np.abs(phi - wphi).max() < 1e-12 * np.abs(wphi).max()


@pytest.mark.parametrize("scale", [1e-3, 0.3, 50.0])
@pytest.mark.parametrize("n,n_leaf", [(2, 1), (33, 1), (400, 2), (397, 7), (400, 32)])
def test_near_pairs_adjoint_of_the_direct_sum(n, n_leaf, scale):
    import torch
    from paper_2502_01496_gb300 import native
    x, m, h = _set(n, scale)
    a_bar = np.random.default_rng(5).normal(size=x.shape)
    f = native.KdFmm(theta=0.0, eps=0.01, n_leaf=n_leaf, soft_kind=native.SOFT_M4, precision=native.FP64)
    f.build(*(torch.tensor(v, device="cuda") for v in (x, m, h))).accel()
    got = [t.cpu().numpy() for t in f.vjp(torch.tensor(a_bar, device="cuda"))]
    for g, w in zip(got, _direct(x, m, h, 0.01, a_bar)):
        assert np.abs(g - w).max() < 1e-12 * np.abs(w).max()
