"""FP64 evaluations of few particles with near lists so long that work items are
groups of segments: the same bits as by segments, and as little memory as with
long ones.  theta = 0 and one particle a leaf: every leaf's near list is all leaves."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _forest(sizes):
    import torch
    ps = [W.plummer(n, 60 + k) for k, n in enumerate(sizes)]
    x = torch.tensor(np.concatenate([p.x for p in ps]), dtype=torch.float64, device="cuda")
    m = torch.tensor(np.concatenate([p.m for p in ps]), dtype=torch.float64, device="cuda")
    return x, m, np.append(0, np.cumsum(sizes))


def _handle(precision):
    from paper_2502_01496_gb300 import native
    return native.KdFmm(theta=0.0, eps=0.01, n_leaf=1, precision=precision)


def test_segments_and_groups_have_the_same_bits():
    """2000 particles have 4e6 near entries, 5e5 segments; three such systems 1.5e6,
    more than the 2^20 that are work items each."""
    import torch
    from paper_2502_01496_gb300 import native
    x, m, off = _forest([2000] * 3)
    f = _handle(native.FP64)
    a, phi = f.build_forest(x, m, None, off).accel()
    for i, j in zip(off, off[1:]):
        g = _handle(native.FP64)
        b, psi = g.build(x[i:j].contiguous(), m[i:j].contiguous()).accel()
        assert torch.equal(a[i:j], b) and torch.equal(phi[i:j], psi)


def test_dense_lists_keep_their_memory():
    """8000 particles, 6.4e7 near entries: beside its lists an FP64 evaluation takes
    no more than a mixed one and a fraction of a byte an entry (128 bytes an entry if
    every segment had its own room); forces and potentials as the direct sum's, to n
    rounding errors of 2^-53 of the sum of the terms' magnitudes, 1e-12."""
    import torch
    from paper_2502_01496_gb300 import native
    n = 8000
    x, m, _ = _forest([n])
    a, phi = torch.empty_like(x), torch.empty_like(m)
    grown = []
    for precision in (native.MIXED, native.FP64):
        f = _handle(precision)
        f.build(x, m)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        f.accel(a, phi)
        torch.cuda.synchronize()
        grown.append(free - torch.cuda.mem_get_info()[0])
        assert f.stats()["nnear"] >= n * (n - 1)
        del f
    assert grown[1] - grown[0] < 4 * n * n, grown
    d = x[:, None, :] - x[None, :, :]
    w = ((d * d).sum(-1) + 0.01 ** 2).rsqrt()
    w.fill_diagonal_(0.0)
    oa, ophi = -torch.einsum("j,ij,ijc->ic", m, w ** 3, d), -(w @ m)
    size = torch.einsum("j,ij->i", m, w ** 3 * d.norm(dim=-1))
    assert ((a - oa).norm(dim=1) < 1e-12 * size).all()
    assert ((phi - ophi).abs() < 1e-12 * ophi.abs()).all()
