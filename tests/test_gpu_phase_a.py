"""Phase A of the build at the particle count where its chunks change size, and
on a handle whose buffers were made for more particles: bit for bit."""
import numpy as np
import pytest

from gpu_common import assert_tree_bit_exact, run_oracle
from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _tree(f, ps):
    import torch
    x, m = (torch.tensor(v, device="cuda") for v in (ps.x, ps.m))
    f.build(x, m)
    return {"ex": f.export(lists=False)}


# 311296 is the last count with chunks of 512; 2049 and 4097 leave one element
# beyond a chunk, 2560 is a whole number of small chunks
def test_phase_a_sizes_on_one_handle(oracle):
    from paper_2502_01496_gb300 import native
    f = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16)
    for n in (311297, 311296, 2049, 2560, 4097, 60013, 400000):
        ps = wl.plummer(n, 60 + n)
        assert_tree_bit_exact(_tree(f, ps), run_oracle(oracle, ps, theta=0.5, n_leaf=16, evaluate=False,
                                                       lists=False))


def test_phase_a_forest(oracle):
    """Segments of very different chunk counts in one level."""
    import torch
    from gpu_common import split_forest
    from paper_2502_01496_gb300 import native
    sizes = [2049, 70000, 3, 2100, 16384, 5000]
    sets = [wl.plummer(n, 70 + n) for n in sizes]
    x = torch.tensor(np.concatenate([p.x for p in sets]), device="cuda")
    m = torch.tensor(np.concatenate([p.m for p in sets]), device="cuda")
    off = np.concatenate([[0], np.cumsum(sizes)])
    f = native.KdFmm(theta=0.5, eps=0.01, n_leaf=8)
    for _ in range(2):                       # followed by the host, then without synchronising
        f.build_forest(x, m, None, off)
        for ex, ps in zip(split_forest(f.export(lists=False), off), sets):
            assert_tree_bit_exact({"ex": ex}, run_oracle(oracle, ps, theta=0.5, n_leaf=8, evaluate=False,
                                                         lists=False))
