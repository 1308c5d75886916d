"""The slot-mode walk with several lanes or a warp per leaf against the thread walk: the
leaf counts where the number of lanes changes, trees smaller than the lanes'
runs, scratch overflow, forests."""
import numpy as np
import pytest

from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _lists(f):
    ex, st = f.export(lists=True), f.stats()
    return [ex.far_off, ex.far_idx, ex.near_off, ex.near_idx], [st[k] for k in ("nfar", "nnear", "np2p", "nexact")]


# leaves of one particle: as many leaves as particles.  A warp serves a leaf up to
# 12160 leaves, 8 lanes to 24320 (on 152 SMs), 4 to 48640, one beyond; theta = 0
# opens every cell and, with 20000 leaves, overflows a lane's scratch of 512 entries
@pytest.mark.parametrize("n,theta", [(1, 0.5), (2, 0.5), (31, 0.5), (33, 0.0), (4000, 0.0), (700, 0.4), (6080, 0.7),
                                     (6081, 0.7), (12160, 0.8), (12161, 0.8), (24321, 0.9), (48641, 1.0), (20000, 0.0)])
def test_split_walk_equals_thread_walk(n, theta, monkeypatch):
    import torch
    from paper_2502_01496_gb300 import native
    ps = wl.plummer(n, 31)
    x, m = (torch.tensor(v, device="cuda") for v in (ps.x, ps.m))
    kw = dict(theta=theta, eps=ps.eps, n_leaf=1)
    f = native.KdFmm(**kw)
    f.build(x, m).accel()
    monkeypatch.setenv("KDFMM_LIST_MODE", "two_pass")       # one thread per leaf, counted and then filled
    g = native.KdFmm(**kw)
    g.build(x, m).accel()
    (a, sa), (b, sb) = _lists(f), _lists(g)
    for u, v in zip(a, b):
        assert np.array_equal(u, v)
    assert sa == sb


def test_split_walk_of_a_forest(monkeypatch):
    import torch
    from paper_2502_01496_gb300 import native
    sizes = [1, 5, 300, 40, 2500]
    sets = [wl.plummer(n, 40 + n) for n in sizes]
    x = torch.tensor(np.concatenate([p.x for p in sets]), device="cuda")
    m = torch.tensor(np.concatenate([p.m for p in sets]), device="cuda")
    off, theta = np.concatenate([[0], np.cumsum(sizes)]), [0.5, 0.3, 0.7, 0.0, 0.6]
    out = []
    for mode in ("", "two_pass"):
        monkeypatch.setenv("KDFMM_LIST_MODE", mode)
        f = native.KdFmm(eps=0.01, n_leaf=4)
        f.build_forest(x, m, None, off, theta=theta).accel()
        out.append(_lists(f))
    for u, v in zip(out[0][0], out[1][0]):
        assert np.array_equal(u, v)
    assert out[0][1] == out[1][1]
