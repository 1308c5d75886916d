"""Mixed near-field kernels with everything near (theta = 0): leaves of 1 to 32
particles fill a staged chunk of 256 sources in every way (32 single-particle
leaves to 8 of 32), their starts on and off the words of the start bitmap.
Softening and supports are wide, so that no pair is close on their scale and the
float32 offsets' error stays small against every term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, 1), (33, 1), (256, 1), (257, 1), (700, 1), (700, 2), (650, 7), (512, 16), (700, 31), (700, 32)]


def _evaluate(x, m, h, n_leaf, eps, kind):
    import torch
    from paper_2502_01496_gb300 import native
    f = native.KdFmm(theta=0.0, eps=eps, n_leaf=n_leaf, soft_kind=kind, precision=native.MIXED)
    f.build(*(None if v is None else torch.tensor(v, device="cuda") for v in (x, m, h)))
    return [t.cpu().numpy() for t in f.accel()]


def _set(n):
    g = np.random.default_rng(3)
    return g.normal(size=(n, 3)), g.uniform(0.5, 1.5, n) / n, g.uniform(0.5, 1.5, n)


# |x| < 4: a pair's offset is off by 14 x 2^-24 a component (the leaf offsets, the
# centres' difference and their sum), 1.5e-6 in all, and its force by 2.5 m times
# that; up to 256 terms are added in float32, 256 x 2^-25 = 7.6e-6 of their
# magnitudes' sum, which is 0.4 (a) and 1 (phi) of the total mass at most; float32
# operations of a term 5e-7.  Together below 1e-5 of the mass, where one misplaced
# source of 700 shows as 5e-4.
@pytest.mark.parametrize("n,n_leaf", SIZES)
def test_plummer_pairs_with_wide_softening(oracle, n, n_leaf):
    x, m, _ = _set(n)
    a, phi = _evaluate(x, m, None, n_leaf, 1.0, 0)
    wa, wphi = oracle.direct(x, m, eps=1.0)
    assert np.abs(a - wa).max() < 1e-5 * m.sum()
    assert np.abs(phi - wphi).max() < 1e-5 * m.sum()


# Supports that hold all pairs (h from 25 to 75): force over distance below
# f = 4/3 / 25^3 a unit of mass and potential below 1.4 / 25.  With the errors above:
# 1.5e-6 + 8e-6 x 7 (the largest distance) of f, 8e-6 of 1.4 / 25.
@pytest.mark.parametrize("n,n_leaf", SIZES)
def test_m4_pairs_with_wide_supports(oracle, n, n_leaf):
    x, m, u = _set(n)
    h = 50.0 * u
    a, phi = _evaluate(x, m, h, n_leaf, 0.01, 1)
    wa, wphi = oracle.direct(x, m, h, soft_kind=1)
    assert np.abs(a - wa).max() < 6e-5 * m.sum() * 4 / 3 / 25 ** 3
    assert np.abs(phi - wphi).max() < 9e-6 * m.sum() * 1.4 / 25
