"""The walk budget counts cells, whoever walks them: a leaf is handed to the
block-wide walk exactly when its walk visits more cells than the budget."""
import pytest

from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget", [1, 63, 64, 65, 200, 1000, 5000])
def test_a_warp_hands_on_the_leaves_that_a_thread_does(budget, monkeypatch):
    """1000 leaves and some: by a warp each in slots, by a thread each in two passes
    (KDFMM_STAT_NHEAVY of the two agree, and the lists' lengths with the default's)."""
    import torch
    from paper_2502_01496_gb300 import native
    ps = wl.plummer(8000, 5)
    x, m = (torch.tensor(v, device="cuda") for v in (ps.x, ps.m))
    out = []
    for mode in ("", "two_pass"):
        monkeypatch.setenv("KDFMM_LIST_MODE", mode)
        f = native.KdFmm(theta=0.4, eps=ps.eps, n_leaf=8)
        native.tree_set_walk_budget(f.handle, budget)
        f.build(x, m).accel()
        out.append(f.stats())
    keys = ("nheavy", "nfar", "nnear", "np2p", "nexact", "nleaves")
    assert [out[0][k] for k in keys] == [out[1][k] for k in keys]
    native.tree_set_walk_budget(f.handle, 0)
    f.build(x, m).accel()
    assert f.stats()["nnear"] == out[0]["nnear"]
