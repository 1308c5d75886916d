"""The FP64 M4 pair at every scale of h and of the separation, coincident
particles among them, against the direct sum in extended precision: forces,
potentials and the adjoint."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


def _side(r, h):
    """(f, g, p) of one side of Eq. 13, q = r/h: force over distance, f'/r, potential."""
    q = r / h
    t = 2 - q
    with np.errstate(all="ignore"):
        F = 1 - t**4 * (1 - L(4) / 5 * t + t**2 / 6)
        f = np.where(q < 1, (L(4) / 3 + q * q * (q / 2 - L(6) / 5)) / h**3, np.where(q < 2, F / r**3, 1 / r**3))
        g = np.where(q < 1, (L(3) / 2 * q - L(12) / 5) / h**5,
                     np.where(q < 2, (t**3 * q**3 - 3 * F) / r**5, -3 / r**5))
        p = np.where(q < 1, (L(7) / 5 + q * q * (-L(2) / 3 + q * q * (L(3) / 10 - q / 10))) / h,
                     np.where(q < 2, (L(8) / 5 + q * q * (-L(4) / 3 + q * (1 + q * (-L(3) / 10 + q / 30)))
                                      - 1 / (15 * q)) / h, 1 / r))
    return f, g, p


def _direct(x, m, h, b):
    """a, phi, x_bar, m_bar and, per value, the sum of its terms' magnitudes."""
    x, m, h, b = (L(v) for v in (x, m, h, b))
    d = x[:, None] - x[None]
    r = np.sqrt((d * d).sum(2))
    (f0, g0, p0), (f1, g1, p1) = _side(r, h[:, None] + 0 * r), _side(r, h[None] + 0 * r)
    f, g, p = (f0 + f1) / 2, (g0 + g1) / 2, (p0 + p1) / 2
    for v in (f, g, p):
        np.fill_diagonal(v, 0)
    db = (d * b[:, None]).sum(2)
    ka = f[..., None] * d
    jb = -f[..., None] * b[:, None] - (g * db)[..., None] * d          # J a_bar_i of pair (i, j)
    jm = f[..., None] * np.abs(b[:, None]) + (np.abs(g) * r * r * np.sqrt((b * b).sum(1))[:, None])[..., None]
    mj = m[None, :, None]
    out = [-(mj * ka).sum(1), -(m * p).sum(1), (mj * jb).sum(1) - (mj * jb).sum(0).reshape(len(m), 3),
           -(f * db).sum(0)]
    mag = [(mj * np.abs(ka)).sum(1), (m * p).sum(1), (mj * jm).sum(1) + (mj * jm).sum(0),
           (f * (np.abs(d) * np.abs(b[:, None])).sum(2)).sum(0)]
    return out, mag


def _check(x, m, h, b, n_leaf):
    """A term takes some 30 float64 operations (each 2^-53; r enters at the fifth
    power at most) and a sum of 40 of them 40 more: below 150 x 2^-53 = 1.7e-14 of
    the magnitudes' sum, which the bound leaves a factor of six."""
    import torch
    from paper_2502_01496_gb300 import native
    t = [torch.tensor(v, dtype=torch.float64, device="cuda") for v in (x, m, h, b)]
    f = native.KdFmm(theta=0.0, eps=0.0, n_leaf=n_leaf, soft_kind=native.SOFT_M4, precision=native.FP64)
    f.build(*t[:3])
    got = [*f.accel(), *f.vjp(t[3])]
    torch.cuda.synchronize()
    out, mag = _direct(x, m, h, b)
    for name, v, want, size in zip(("a", "phi", "x_bar", "m_bar"), got, out, mag):
        v = v.cpu().numpy()
        assert np.isfinite(v).all(), name
        assert (np.abs(v - want) <= 1e-13 * size).all(), (name, np.max(np.abs(v - want) / (size + (size == 0))))


@pytest.mark.parametrize("n,n_leaf", [(2, 32), (2, 1), (40, 32), (40, 7)])
@pytest.mark.parametrize("h", [1e-30, 1e-24, 1e-23, 1e-20, 1e-19, 1e-10, 0.4, 1e18, 1e20, 1e25])
def test_m4_pairs_for_every_h(n, n_leaf, h):
    """The first fifth of 40 particles (both of two) lie in one place each with a
    partner; h within a factor of two of the given one."""
    rng = np.random.default_rng(n + n_leaf)
    x = rng.normal(size=(n, 3))
    k = max(n // 5, 1)
    x[k:2 * k] = x[:k]
    _check(x, rng.uniform(0.5, 1.5, n), h * rng.uniform(0.7, 1.4, n), rng.normal(size=(n, 3)), n_leaf)


@pytest.mark.parametrize("n_leaf", [1, 32])
@pytest.mark.parametrize("h", [1e-50, 1e-3, 1e30])
@pytest.mark.parametrize("power", [-48.0, -40.0, -19.5, -18.5, -10.0, 0.0, 10.0, 18.5, 19.5, 40.0, 48.0])
def test_m4_pair_for_every_separation(power, h, n_leaf):
    """Two particles; 1/r over its range (r^-5 stays a normal number)."""
    rng = np.random.default_rng(7)
    x = np.zeros((2, 3))
    x[1] = 10.0 ** power * rng.uniform(0.3, 1.0, 3)
    _check(x, np.array([0.7, 1.3]), h * np.array([1.0, 1.5]), rng.normal(size=(2, 3)), n_leaf)
