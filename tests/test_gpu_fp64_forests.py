"""FP64 evaluations at the limits of the P2P segment lengths (8192, 65536 and
262144 particles of a system), alone and in forests on both sides of the size
from which work items are groups of segments: the same bits, and little memory."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _systems(sizes, soft):
    ps = [W.plummer(n, 40 + k) if soft == "plummer" else W.polytrope_binary(n // 2, 40 + k)
          for k, n in enumerate(sizes)]
    off = np.append(0, np.cumsum([p.n for p in ps]))
    return ps, off


def _cuda(v):
    import torch
    return torch.tensor(v, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("soft", ["plummer", "m4"])
@pytest.mark.parametrize("sizes", [[100, 8190, 8192, 20000], [8190, 300, 8192, 65534, 65536, 120000],
                                   [262142, 1000], [262144, 1000]])
def test_a_system_has_the_same_bits_alone_and_in_a_forest(sizes, soft):
    """36482, 267418 and some 263000 particles: segments as work items below 262144
    particles in all, groups of them above."""
    import torch
    from paper_2502_01496_gb300 import native
    ps, off = _systems(sizes, soft)
    kind = native.SOFT_PLUMMER if soft == "plummer" else native.SOFT_M4
    pars = dict(theta=0.7, eps=0.01, n_leaf=16, soft_kind=kind, precision=native.FP64)
    h = None if soft == "plummer" else _cuda(np.concatenate([p.h for p in ps]))
    f = native.KdFmm(**pars)
    f.build_forest(_cuda(np.concatenate([p.x for p in ps])), _cuda(np.concatenate([p.m for p in ps])), h, off)
    a, phi = f.accel()
    for p, i, j in zip(ps, off, off[1:]):
        g = native.KdFmm(**pars)
        b, psi = g.build(_cuda(p.x), _cuda(p.m), None if h is None else _cuda(p.h)).accel()
        assert torch.equal(a[i:j], b) and torch.equal(phi[i:j], psi), (i, j)


@pytest.mark.parametrize("n", [8191, 8192, 65535, 65536, 262143, 262144])
def test_segment_limits_against_the_oracle(oracle, n):
    """Every 50th leaf; the bound of the FP64 parity tests."""
    import torch
    from paper_2502_01496_gb300 import native
    p = W.plummer(n, 50)
    f = native.KdFmm(theta=0.7, eps=p.eps, n_leaf=16, precision=native.FP64)
    a, phi = f.build(_cuda(p.x), _cuda(p.m)).accel()
    T = oracle.Tree(p.x, p.m, None, theta=0.7, n_leaf=16, eps=p.eps)
    cells = T.cells()
    leaves = np.nonzero(cells.left < 0)[0][::50]
    oa, ophi = T.eval_threads(leaves=leaves)
    rows = np.isfinite(ophi)
    torch.cuda.synchronize()
    a, phi = a.cpu().numpy()[rows], phi.cpu().numpy()[rows]
    assert rows.sum() > 100
    assert (np.linalg.norm(a - oa[rows], axis=1) < 1e-12 * np.linalg.norm(oa[rows], axis=1)).all()
    assert (np.abs(phi - ophi[rows]) < 1e-12 * np.abs(ophi[rows])).all()


def test_a_forest_of_small_systems_keeps_its_memory():
    """256 systems of 4096: what an FP64 evaluation allocates beside its lists is a
    fraction of a byte a near entry more than a mixed one (1 KB per 256 entries
    each; 128 bytes an entry when every short segment had its own room)."""
    import torch
    from paper_2502_01496_gb300 import native
    ps, off = _systems([4096] * 256, "plummer")
    x, m = _cuda(np.concatenate([p.x for p in ps])), _cuda(np.concatenate([p.m for p in ps]))
    a, phi = torch.empty_like(x), torch.empty_like(m)
    grown = []
    for precision in (native.MIXED, native.FP64):
        f = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16, precision=precision)
        f.build_forest(x, m, None, off)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        f.accel(a, phi)
        torch.cuda.synchronize()
        grown.append(free - torch.cuda.mem_get_info()[0])
        near = f.stats()["nnear"]
        del f
    assert grown[1] - grown[0] < 4 * near, (grown, near)
