"""The sums of the mixed adjoint's P2P reverse keep float64: terms that float32
forms and float64 adds without rounding come out exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OWN, NEAR, FAR = (0.0, 0.0, 0.0), (0.5, 0.25, 1.0), (128.0, 96.0, -64.0)


def _adjoint(near, far, b_own, b_other, n_leaf):
    """x_bar and m_bar of the particle at the origin, with `near` and `far` others in
    one place each (coordinates on which every difference is exact)."""
    import torch
    from paper_2502_01496_gb300 import native
    x = np.array([OWN] + [NEAR] * near + [FAR] * far)
    b = np.array([b_own] + [b_other] * (near + far))
    cuda = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")
    f = native.KdFmm(theta=0.0, eps=0.5, n_leaf=n_leaf, precision=native.MIXED)
    f.build(cuda(x), cuda(np.ones(len(x)))).accel()
    x_bar, m_bar = f.vjp(cuda(b))
    return np.append(x_bar[0].cpu().numpy(), m_bar[0].cpu().numpy())


# A term of the far place is some 2^-13 to 2^-23 of one of the near place.  Terms are
# multiples of their own last float32 bit, so float64 adds them without rounding, in
# any order, if the sum in units of the smaller term's last bit stays below 2^53
# (asserted), where two float32 numbers lose bits past 2^48.
# Source side: one target a leaf (a leaf's terms are added in float32).
@pytest.mark.parametrize("near,far", [(64, 1003), (5, 700), (1, 31), (64, 2)])
@pytest.mark.parametrize("side,n_leaf", [("target", 1), ("target", 5), ("target", 32), ("source", 1)])
def test_sums_are_exact(side, n_leaf, near, far):
    b = (0.75, -1.5, 0.375)
    own, other = (b, (0.0,) * 3) if side == "target" else ((0.0,) * 3, b)
    one_near, one_far = _adjoint(1, 0, own, other, 1), _adjoint(0, 1, own, other, 1)
    got = _adjoint(near, far, own, other, n_leaf)
    assert (np.abs(one_near[:3]) > 0).all() and (np.abs(one_far[:3]) > 0).all()
    last_bit = 2.0 ** (np.floor(np.log2(np.minimum(np.abs(one_near), np.abs(one_far)) + 1e-300)) - 23)
    assert ((near * np.abs(one_near) + far * np.abs(one_far))[:3] / last_bit[:3] < 2.0 ** 53).all()
    assert np.array_equal(got, near * one_near + far * one_far)
