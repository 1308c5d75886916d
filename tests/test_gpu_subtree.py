"""The shared-memory subtrees at the edges of their octets, batches and cells:
the tree equals the oracle's bit for bit."""
import numpy as np
import pytest

from gpu_common import assert_tree_bit_exact, oracle_cell_arrays, run_gpu, run_oracle
from paper_2502_01496_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


# one subtree of up to 2048 particles; octets of 8, batches of 128 cells (leaves
# of 1 make levels of up to ~1000 cells), the first sizes that need phase A
@pytest.mark.parametrize("n,n_leaf", [(2, 1), (7, 1), (8, 1), (9, 3), (33, 32), (64, 8), (65, 1), (1023, 1),
                                      (1024, 5), (2047, 1), (2048, 1), (2048, 16), (2049, 1), (4099, 2)])
def test_subtree_sizes(oracle, n, n_leaf):
    ps = wl.plummer(n, 50 + n)
    kw = dict(theta=0.5, n_leaf=n_leaf)
    g = run_gpu(ps, precision=0, lists=False, **kw)
    assert_tree_bit_exact(g, run_oracle(oracle, ps, evaluate=False, lists=False, **kw))


# boxes whose longest axis the float32 box cannot tell (a cubic lattice, equal
# extents; coordinates far from the origin), and cells that no cut divides.
# Everything that decides the tree is compared; the quadrupoles are left out,
# whose rounding scales with |x|, which is 10^8 sizes in "far", and not with the
# size, which is 0 in "coincident"
@pytest.mark.parametrize("case", ["lattice", "far", "coincident", "line"])
def test_subtree_boxes(oracle, case):
    rng = np.random.default_rng(3)
    if case == "lattice":
        g = np.arange(12) / 12.0
        x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    elif case == "far":
        x = 1e6 + 1e-2 * rng.normal(size=(1500, 3))
    elif case == "coincident":
        x = np.repeat(rng.normal(size=(6, 3)), 200, axis=0)
    else:
        x = np.zeros((999, 3))
        x[:, 1] = rng.normal(size=999)
    ps = wl.ParticleSet(x=x, m=rng.uniform(0.5, 1.0, len(x)), h=None, soft_kind=0, eps=0.01, name=case)
    kw = dict(theta=0.5, n_leaf=4)
    ex = run_gpu(ps, precision=0, lists=False, **kw)["ex"]
    o = run_oracle(oracle, ps, evaluate=False, lists=False, **kw)
    ints, reals = oracle_cell_arrays(o["cells"])
    assert np.array_equal(ex.perm, o["order"])
    assert np.array_equal(ex.cell_ints, ints)
    assert np.array_equal(ex.cell_reals[:, :6], reals[:, :6])
