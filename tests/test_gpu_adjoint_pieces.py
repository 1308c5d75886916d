"""Near lists and transposed near lists of the adjoint just below, at and above one
work item (8 entries in a small call, 256 in one whose lists fill the GPU)."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as wl
from test_gpu_adjoint_lists import _direct

pytestmark = pytest.mark.gpu


# theta = 0 and leaves of one: a list has as many entries as its system has
# particles.  One system of 7 to 17: items of 8; 29 of 255 to 257: some 1.9e6
# entries, which makes 12 warps a scheduler with items of 256.
@pytest.mark.parametrize("n_sys,n", [(1, 7), (1, 8), (1, 9), (1, 16), (1, 17), (29, 255), (29, 256), (29, 257)])
@pytest.mark.parametrize("kind", ["plummer", "m4"])
# as for other direct sums: float64 sums 1e-12 of the largest component; mixed 1e-5
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_lists_around_one_item(kind, n_sys, n, precision, tol):
    import torch
    from paper_2502_01496_gb300 import native
    ps = [wl.plummer(n, 60 + k) for k in range(n_sys)]
    rng = np.random.default_rng(8)
    h = [rng.uniform(0.05, 0.5, n) for _ in ps] if kind == "m4" else None
    b = rng.normal(size=(n_sys * n, 3))
    cuda = lambda v: torch.tensor(v, device="cuda")
    f = native.KdFmm(theta=0.0, eps=0.05, n_leaf=1, precision=precision,
                     soft_kind=native.SOFT_M4 if h else native.SOFT_PLUMMER)
    f.build_forest(cuda(np.concatenate([p.x for p in ps])), cuda(np.concatenate([p.m for p in ps])),
                   cuda(np.concatenate(h)) if h else None, np.arange(n_sys + 1) * n).accel()
    x_bar, m_bar = (t.cpu().numpy() for t in f.vjp(cuda(b)))
    for k, p in enumerate(ps):
        s = slice(k * n, (k + 1) * n)
        for got, want in zip((x_bar[s], m_bar[s]), _direct(p.x, p.m, h[k] if h else None, 0.05, b[s])):
            assert np.abs(got - want).max() < tol * np.abs(want).max(), k
