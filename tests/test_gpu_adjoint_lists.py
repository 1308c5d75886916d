"""The P2P reverse over transposed near lists at the sizes of its splits: leaves
of 1 to 32 particles (one lane to a whole warp per source, every depth of the
per-leaf tree sum), and source lists below, at and above one work item."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _direct(x, m, h, eps, a_bar):
    """(x_bar, m_bar) of the direct sum by plain float64 autograd on the CPU."""
    import torch
    x = torch.tensor(x, requires_grad=True)
    m = torch.tensor(m, requires_grad=True)
    d = x[:, None] - x[None]
    r2 = (d * d).sum(-1) + torch.eye(len(x), dtype=torch.float64)     # no 0 / 0 on the diagonal
    if h is None:
        f = (r2 + eps * eps) ** -1.5
    else:
        r = r2.sqrt()

        def side(hh):
            q = r / hh
            inner = (4 / 3 + q * q * (-1.2 + 0.5 * q)) / hh ** 3
            outer = (8 / 3 - 3 * q + 1.2 * q ** 2 - q ** 3 / 6 - 1 / (15 * q ** 3)) / hh ** 3
            return torch.where(q < 1, inner, torch.where(q < 2, outer, r ** -3))

        ht = torch.tensor(h)
        f = 0.5 * (side(ht[:, None]) + side(ht[None]))
    f = f * (1 - torch.eye(len(x), dtype=torch.float64))
    a = -(m[None, :, None] * f[..., None] * d).sum(1)
    g = torch.autograd.grad(a, (x, m), torch.tensor(a_bar))
    return [t.numpy() for t in g]


# theta = 0 opens everything: every leaf is near every other, so a source list
# has as many entries as there are leaves.  500 particles in leaves of 1 and 3
# give lists of several work items (128 entries each), larger leaves one.
@pytest.mark.parametrize("n_leaf", [1, 3, 5, 9, 17, 32])
@pytest.mark.parametrize("kind", ["plummer", "m4"])
# float64 sums of 500 terms: 1e-12 of the largest component; mixed: float32
# terms (6e-8) with cancellations inside a pair: 1e-5
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_adjoint_of_the_direct_sum(kind, n_leaf, precision, tol):
    import torch
    from paper_2502_01496_gb300 import native
    ps = wl.plummer(500, 21) if kind == "plummer" else wl.polytrope_binary(250, 21)
    a_bar = np.random.default_rng(5).normal(size=ps.x.shape)
    cuda = lambda v: None if v is None else torch.tensor(v, device="cuda")
    f = native.KdFmm(theta=0.0, eps=ps.eps, n_leaf=n_leaf, soft_kind=ps.soft_kind, precision=precision)
    f.build(cuda(ps.x), cuda(ps.m), cuda(ps.h)).accel()
    got = [t.cpu().numpy() for t in f.vjp(cuda(a_bar))]
    want = _direct(ps.x, ps.m, ps.h, ps.eps, a_bar)
    for g, w in zip(got, want):
        assert np.abs(g - w).max() < tol * np.abs(w).max()
