"""Builds that outgrow what was launched for them: a kept handle whose next tree
needs more levels than its last one, alone or as a replayed graph, and forests
with more segments than the lists hold."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 20000


def _uniform(rng):
    return rng.uniform(-1.0, 1.0, (N, 3))


def _steep(rng):
    """Radii over twelve decades in one octant: a cut through the centre of mass
    takes an eighth of the particles off, so 20000 need some 18 levels down to
    cells of 2048, where a uniform set needs 4."""
    return 10.0 ** rng.uniform(-12.0, 0.0, (N, 1)) * rng.uniform(0.9, 1.1, (N, 3))


@pytest.mark.parametrize("call", ["build", "batch"])
@pytest.mark.parametrize("precision", [0, 1])
def test_a_tree_with_more_levels_than_the_last_one(call, precision):
    """Same number of particles and same buffers, uniform and then steep: bit for
    bit the results of a fresh handle."""
    import torch
    from paper_2502_01496_gb300 import native
    rng = np.random.default_rng(5)
    x = torch.tensor(_uniform(rng), device="cuda")
    m = torch.full((N,), 1.0 / N, dtype=torch.float64, device="cuda")
    a, phi = torch.empty_like(x), torch.empty_like(m)
    steep = torch.tensor(_steep(rng), device="cuda")
    pars = dict(theta=0.5, eps=1e-3, n_leaf=16, precision=precision)
    kept = native.KdFmm(**pars)

    def evaluate():
        if call == "build":
            kept.build(x, m).accel(a, phi)
        else:
            native.fmm_accel_batched(kept.handle, x, m, None, np.array([0, N // 4, N]), kept.params, a, phi)

    for _ in range(3):                    # (batch: eager, captured, replayed)
        evaluate()
    x.copy_(steep)
    evaluate()
    fresh = native.KdFmm(**pars)
    b, psi = torch.empty_like(x), torch.empty_like(m)
    if call == "build":
        fresh.build(steep, m).accel(b, psi)
    else:
        native.fmm_accel_batched(fresh.handle, steep, m, None, np.array([0, N // 4, N]), fresh.params, b, psi)
    torch.cuda.synchronize()
    assert torch.isfinite(a).all()
    assert torch.equal(a, b) and torch.equal(phi, psi)


def test_a_forest_of_single_particles_is_refused():
    """More root leaves than the list of leaf segments (n / 4 + 64) holds."""
    import torch
    from paper_2502_01496_gb300 import native
    rng = np.random.default_rng(6)
    x = torch.tensor(rng.uniform(-1.0, 1.0, (4000, 3)), device="cuda")
    m = torch.ones(4000, dtype=torch.float64, device="cuda")
    f = native.KdFmm(theta=0.5, eps=0.1, n_leaf=16, precision=native.FP64)
    for _ in range(2):
        with pytest.raises(native.KdfmmError) as e:
            f.build_forest(x, m, None, np.arange(4001))
        assert "capacity" in str(e.value)
    a, _ = f.build_forest(x, m, None, np.array([0, 1000, 4000])).accel()
    assert torch.isfinite(a).all()
