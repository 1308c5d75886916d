"""The library's own reciprocal root and conversions over their exponents, seen
through systems of two particles: leaves of one, theta = 0, no softening, so a
particle's potential is -m / r of the other one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _potentials(precision, x, m):
    """phi of the particle at the origin of each system; the other, of mass m, at (x, 0, 0)."""
    import torch
    from paper_2502_01496_gb300 import native
    n = len(x)
    pos = np.zeros((2 * n, 3))
    pos[1::2, 0] = x
    mass = np.ones(2 * n)
    mass[1::2] = m
    f = native.KdFmm(theta=0.0, eps=0.0, n_leaf=1, precision=precision)
    f.build_forest(torch.tensor(pos, device="cuda"), torch.tensor(mass, device="cuda"), None,
                   np.arange(0, 2 * n + 1, 2))
    _, phi = f.accel()
    torch.cuda.synchronize()
    return phi.cpu().numpy()[::2]


def _mantissas(rng, n):
    """In [1, 2): random ones, the ends, and float32 values with the ties above them."""
    f32 = rng.integers(0, 1 << 23, n) * 2.0 ** -23
    kind = rng.integers(0, 5, n)
    return 1.0 + np.choose(kind, [rng.uniform(0, 1, n), np.zeros(n), np.full(n, 1 - 2.0 ** -52), f32,
                                  f32 + 2.0 ** -24])


def test_reciprocal_root_within_half_a_unit():
    """rsqrt64 of r^2 from 2^-1000 to 2^1000: 0.501 units in the last place by its
    derivation (the reference is off by 0.001 at most)."""
    rng = np.random.default_rng(1)
    x = _mantissas(rng, 40000) * 2.0 ** rng.integers(-500, 500, 40000)
    phi = _potentials(0, x, 1.0)
    want = 1 / np.sqrt(np.longdouble(x * x))
    unit = np.spacing(want.astype(np.float64))
    assert (np.abs(-phi - want) <= 0.503 * unit).all(), np.max(np.abs(-phi - want) / unit)


def test_masses_round_to_nearest_float():
    """Mixed mode takes m as the nearest float32 (ties to even), subnormal ones
    included: phi is its product with the reciprocal distance, 1 here."""
    rng = np.random.default_rng(2)
    m = np.append(1.0, _mantissas(rng, 40000) * 2.0 ** rng.integers(-148, 126, 40000))
    phi = -_potentials(1, np.ones(len(m)), m)
    inv = np.float32(phi[0])
    assert abs(inv - 1) <= 2.0 ** -22
    assert np.array_equal(phi, (m.astype(np.float32) * inv).astype(np.float64))


def test_centres_keep_their_high_and_low_parts():
    """Mixed distances between single-particle leaves come from (high, low) float32
    centres: phi within the approximate root (2^-22.4) and four roundings (2^-24)."""
    rng = np.random.default_rng(3)
    x = _mantissas(rng, 40000) * 2.0 ** rng.integers(-55, 55, 40000)
    phi = -_potentials(1, x, 1.0)
    assert (np.abs(phi * x - 1) <= 2.0 ** -21).all(), np.max(np.abs(phi * x - 1))
