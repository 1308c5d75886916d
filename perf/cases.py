"""Performance cases of the kd-tree FMM: what its users have it do, over the range of sizes and options.

Every case goes through the public entry points (``native.KdFmm``, ``native.fmm_accel_batched``,
``native.total_momentum``, ``dynamics.fmm_accel`` with autograd, ``dynamics.leapfrog``).  Particle sets follow the
recipes of ``paper_2502_01496_gb300/workloads.py`` (Plummer spheres, binaries of n = 1 polytropes, uniform +
clumps), drawn on the GPU.  ``exact`` restates the method in float64 numpy and torch, without the package's code.
"""
import math
import random

import numpy as np
import torch

from paper_2502_01496_gb300 import dynamics, native

F64 = torch.float64


def listed():
    return [
        # the smallest call: a thousand particles (a small cluster, a unit test, one star of a toy run); launches and
        # host round trips are all of it
        {"name": "step_plummer_1009_mixed", "do": "step", "set": "plummer", "n": 1009, "theta": 0.5, "n_leaf": 16,
         "precision": "mixed"},
        # the plain method: one float64 evaluation of 4096 particles, checked against the direct sum by its users
        {"name": "step_plummer_4096_fp64", "do": "step", "set": "plummer", "n": 4096, "theta": 0.5, "n_leaf": 16,
         "precision": "fp64"},
        # an ordinary single cluster of odd size with a smaller leaf
        {"name": "step_plummer_60013_mixed", "do": "step", "set": "plummer", "n": 60013, "theta": 0.6, "n_leaf": 12,
         "precision": "mixed"},
        # an accurate float64 evaluation (small theta) of a neutron-star binary, the size of the drift study's runs
        {"name": "step_binary_32770_fp64", "do": "step", "set": "binary", "n": 32770, "theta": 0.3, "n_leaf": 16,
         "precision": "fp64"},
        # the benchmark's workload: build + evaluation + total force of the 2 x 2^20 binary, in both precisions
        {"name": "step_binary_2097152_mixed", "do": "step", "set": "binary", "n": 2097152, "theta": 0.5, "n_leaf": 16,
         "precision": "mixed"},
        {"name": "step_binary_2097152_fp64", "do": "step", "set": "binary", "n": 2097152, "theta": 0.5, "n_leaf": 16,
         "precision": "fp64"},
        # the large single evaluation: 2^24 particles, half uniform and half in clumps, leaves of up to 32
        {"name": "step_clumps_16777216_mixed", "do": "step", "set": "clumps", "n": 16777216, "theta": 0.5,
         "n_leaf": 32, "precision": "mixed"},
        # serving: 256 independent systems of uneven size and theta in one call, repeated on the same buffers
        {"name": "batch_256_mixed", "do": "batch", "systems": 256, "n_min": 2048, "n_max": 262144, "layout": 1,
         "n_leaf": 16, "precision": "mixed"},
        # differentiation: accelerations and their gradients with respect to positions and masses
        {"name": "grad_plummer_1048576_mixed", "do": "grad", "set": "plummer", "n": 1048576, "theta": 0.5,
         "n_leaf": 16, "precision": "mixed"},
        {"name": "grad_binary_16386_fp64", "do": "grad", "set": "binary", "n": 16386, "theta": 0.5, "n_leaf": 16,
         "precision": "fp64"},
        # the momentum-conserving variant (symmetric dual walk) on a binary
        {"name": "dual_binary_262146_mixed", "do": "dual", "set": "binary", "n": 262146, "theta": 0.5, "n_leaf": 16,
         "precision": "mixed"},
        # a whole call: four steps of the differentiable integrator with checkpoints, and the gradient of the final
        # centre-of-mass displacement
        {"name": "leapfrog_plummer_20011_mixed", "do": "leapfrog", "set": "plummer", "n": 20011, "theta": 0.5,
         "n_leaf": 16, "precision": "mixed", "steps": 4, "every": 2},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    do = rng.choice(["step", "step", "step", "step", "batch", "grad", "grad", "dual", "leapfrog"])
    precision = rng.choice(["mixed", "mixed", "fp64"]) if do in ("step", "grad") else "mixed"
    # leaf sizes up to the usual 16: the gradient's pooled handles outlive their call, and no other handle in the
    # process may then build with larger leaves than theirs
    case = {"do": do, "precision": precision, "n_leaf": rng.choice([8, 12, 16, 16]) if do in ("step", "batch") else 16}
    if do == "batch":
        lo = _log_uniform(rng, 1000, 8000)
        return case | {"systems": _log_uniform(rng, 3, 128), "n_min": lo, "n_max": lo * rng.choice([4, 16, 64]),
                       "layout": rng.randrange(1 << 20)}
    kind = rng.choice(["plummer", "binary", "clumps"])
    top = {"step": 6000000, "grad": 700000, "dual": 1000000, "leapfrog": 60000}[do]
    if precision == "fp64":
        top = {"step": 1000000, "grad": 100000}[do]
    n = _log_uniform(rng, 1000, top)
    case |= {"set": kind, "n": n + n % 2 if kind == "binary" else n, "theta": round(rng.uniform(0.3, 0.9), 3)}
    if do == "leapfrog":
        case |= {"steps": rng.randint(2, 6), "every": rng.randint(1, 3)}
    return case


# --- particle sets ----------------------------------------------------------------------------------------------

EPS = {"plummer": 0.01, "binary": 0.0, "clumps": 1e-3}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=F64)


def _isotropic(g, n):
    cz, ph = _uniform(g, n, lo=-1.0), _uniform(g, n, hi=2.0 * math.pi)
    sz = torch.sqrt(1.0 - cz * cz)
    return torch.stack([sz * torch.cos(ph), sz * torch.sin(ph), cz], 1)


def _plummer(g, n):
    r = 1.0 / torch.sqrt(_uniform(g, n, lo=1e-12, hi=0.999) ** (-2.0 / 3.0) - 1.0)
    return r[:, None] * _isotropic(g, n), torch.full((n,), 1.0 / n, device="cuda", dtype=F64), None


def _polytrope(g, n):
    """An n = 1 polytrope of radius and mass 1: a jittered lattice ball, stretched to the enclosed-mass profile."""
    a = (4.0 * math.pi / (3.0 * n)) ** (1.0 / 3.0)
    k = math.ceil(1.0 / a) + 2
    axis = torch.arange(-k, k + 1, device="cuda", dtype=F64) * a
    lat = torch.cartesian_prod(axis, axis, axis)
    p = lat[torch.sort(lat.square().sum(1), stable=True).indices[:n]]
    p = p + _uniform(g, n, 3, lo=-0.1 * a, hi=0.1 * a)
    ru = p.norm(dim=1)
    rank = torch.empty(n, device="cuda", dtype=F64)
    rank[torch.sort(ru, stable=True).indices] = torch.arange(n, device="cuda", dtype=F64)
    frac = (rank + 0.5) / n
    lo, hi = torch.zeros_like(frac), torch.full_like(frac, math.pi)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        below = (torch.sin(mid) - mid * torch.cos(mid)) / math.pi < frac
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    xi = 0.5 * (lo + hi)
    x = p * (xi / math.pi / ru)[:, None]
    rho = 0.25 * math.pi * torch.clamp(torch.sin(xi) / xi, min=0.01)
    return x, torch.full((n,), 1.0 / n, device="cuda", dtype=F64), 1.2 * (1.0 / n / rho) ** (1.0 / 3.0)


def _binary(g, n):
    stars = [_polytrope(g, n // 2), _polytrope(g, n // 2)]
    for sign, (x, _, _) in zip((-2.0, 2.0), stars):
        x[:, 0] += sign
    return tuple(torch.cat(t).contiguous() for t in zip(*stars))


def _clumps(g, n):
    nc = n - n // 2
    centres = _uniform(g, 64, 3)
    which = torch.arange(nc, device="cuda") % 64
    xc = centres[which] + 0.01 * torch.randn(nc, 3, generator=g, device="cuda", dtype=F64)
    m = torch.exp(_uniform(g, n, hi=math.log(10.0)))
    return torch.cat([_uniform(g, n // 2, 3), xc]), m / m.sum(), None


_SETS = {"plummer": _plummer, "binary": _binary, "clumps": _clumps}


def _layout(case):
    """Sizes and opening parameters of a batch's systems: part of the case, not of its inputs."""
    rng = random.Random(case["layout"])
    sizes = [_log_uniform(rng, case["n_min"], case["n_max"]) for _ in range(case["systems"])]
    return sizes, [rng.uniform(0.3, 1.0) for _ in sizes]


def _inputs(case, seed):
    g = _gen(seed)
    if case["do"] == "batch":
        x, m, _ = _plummer(g, sum(_layout(case)[0]))
        m = torch.cat([torch.full((k,), 1.0 / k, device="cuda", dtype=F64) for k in _layout(case)[0]])
        return {"x": x, "m": m, "h": None}
    x, m, h = _SETS[case["set"]](g, case["n"])
    d = {"x": x, "m": m, "h": h}
    if case["do"] == "grad":
        d["a_bar"] = torch.randn(case["n"], 3, generator=g, device="cuda", dtype=F64)
    if case["do"] == "leapfrog":
        # isotropic velocities at a Plummer sphere's dispersion, sigma^2 = 1 / (6 sqrt(1 + r^2))
        sigma = (6.0 * torch.sqrt(1.0 + x.square().sum(1))) ** -0.5
        d["v"] = sigma[:, None] * torch.randn(case["n"], 3, generator=g, device="cuda", dtype=F64)
    return d


def _params(case):
    kind = case.get("set", "plummer")
    return dict(theta=case.get("theta", 0.5), eps=EPS[kind], n_leaf=case["n_leaf"],
                soft_kind=native.SOFT_M4 if kind == "binary" else native.SOFT_PLUMMER,
                precision=native.FP64 if case["precision"] == "fp64" else native.MIXED,
                walk=native.WALK_DUAL if case["do"] == "dual" else native.WALK_LEAF)


# --- one pass ---------------------------------------------------------------------------------------------------

def prepare(case, seed):
    """The particles, and what a program keeps between evaluations: its handle and its output arrays."""
    s = dict(_inputs(case, seed), case=case, params=_params(case))
    n = s["x"].shape[0]
    if case["do"] in ("grad", "leapfrog"):
        s["x"].requires_grad_(True)
        if case["do"] == "grad":
            s["m"].requires_grad_(True)
        return s
    s["f"] = native.KdFmm(**s["params"])
    s["a"] = torch.empty(n, 3, device="cuda", dtype=F64)
    s["phi"] = torch.empty(n, device="cuda", dtype=F64)
    s["force"] = torch.empty(3, device="cuda", dtype=F64)
    if case["do"] == "batch":
        sizes, theta = _layout(case)
        s["offsets"] = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        s["theta"] = np.array(theta)
        s["leaf"] = np.full(len(sizes), case["n_leaf"], dtype=np.int32)
        s["eps"] = np.full(len(sizes), EPS["plummer"])
    return s


def run(s):
    do = s["case"]["do"]
    if do == "grad":
        a = dynamics.fmm_accel(s["x"], s["m"], s["h"], **s["params"])
        x_bar, m_bar = torch.autograd.grad(a, (s["x"], s["m"]), s["a_bar"])
        return {"a": a, "x_bar": x_bar, "m_bar": m_bar}
    if do == "leapfrog":
        x, v, a = dynamics.leapfrog(s["x"], s["v"], s["m"], s["h"], steps=s["case"]["steps"], dt=1e-3,
                                    checkpoint_every=s["case"]["every"], **s["params"])
        shift = dynamics.centre_of_mass(x, s["m"]) - dynamics.centre_of_mass(s["x"], s["m"])
        s["x"].grad = None
        shift.square().sum().backward()
        return {"x": x, "v": v, "a": a, "x_bar": s["x"].grad}
    if do == "batch":
        native.fmm_accel_batched(s["f"].handle, s["x"], s["m"], None, s["offsets"], s["f"].params, s["a"], s["phi"],
                                 theta=s["theta"], eps=s["eps"], n_leaf=s["leaf"])
        return {"a": s["a"], "phi": s["phi"]}
    s["f"].build(s["x"], s["m"], s["h"])
    s["f"].accel(s["a"], s["phi"])
    if do == "dual":                     # its total force is rounding alone
        return {"a": s["a"], "phi": s["phi"]}
    native.total_momentum(s["m"], s["a"], s["force"])
    return {"a": s["a"], "phi": s["phi"], "force": s["force"]}


# Interactions per particle at theta = 0.5 and leaves of up to 16, counted on the sets above at 1 to 2 million
# particles: (pairs summed directly, cells expanded into a leaf divided by its particles).
_COUNTS = {"plummer": (1120.0, 126.0), "binary": (735.0, 32.0), "clumps": (421.0, 29.0)}


def work(case):
    """Bytes: the caller's arrays, read or written once.  Operations: 20 (Plummer) or 30 (M4) per direct pair and 250
    per expansion, with the pair counts of ``_COUNTS`` scaled to theta and the leaf size; a gradient costs twice
    its evaluation more."""
    if case["do"] == "batch":
        sizes, theta = _layout(case)
        n, th, kind = sum(sizes), sum(theta) / len(theta), "plummer"
    else:
        n, th, kind = case["n"], case["theta"], case["set"]
    pairs, far = _COUNTS[kind]
    pairs = min(n - 1.0, pairs * case["n_leaf"] / 16.0 * (1.0 if kind == "binary" else (0.5 / th) ** 2))
    far *= 16.0 / case["n_leaf"] * (0.5 / th) ** 2
    flops = n * (pairs * (30.0 if kind == "binary" else 20.0) + far * 250.0)
    per = 32 + 8 * (kind == "binary")                          # x, m and h
    if case["do"] == "grad":
        return {"bytes": float(n * (per + 24 + 24 + 32)), "flops": 3.0 * flops}
    if case["do"] == "leapfrog":
        return {"bytes": float(n * (per + 24 + 4 * 24)), "flops": (3.0 * case["steps"] + 1.0) * flops}
    return {"bytes": float(n * (per + 32)), "flops": flops}


# --- the method in 64 bits, plainly -----------------------------------------------------------------------------

def _pairwise(v):
    """Sum over the rows as a perfect binary tree, padded with zeros to a power of two."""
    size = 1 << max(0, (len(v) - 1).bit_length())
    v = np.concatenate([v, np.zeros((size - len(v),) + v.shape[1:])])
    while len(v) > 1:
        v = v[0::2] + v[1::2]
    return v[0]


def _tree(x, m, h, n_leaf):
    """Cells in pre-order: (particles in caller order, centre of mass, size, largest h, left, right)."""
    cells = []

    def grow(idx):
        me = len(cells)
        p = x[idx]
        mass = _pairwise(m[idx])
        com = _pairwise(m[idx, None] * p) / mass
        d = p - com
        size = math.sqrt(((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]).max())
        cells.append([idx, com, size, h[idx].max(), -1, -1])
        if len(idx) > n_leaf:
            axis = int(np.argmax(p.max(0) - p.min(0)))
            left = p[:, axis] < com[axis]
            if left.all() or not left.any():
                left = np.arange(len(idx)) < len(idx) // 2
            cells[me][4] = grow(idx[left])
            cells[me][5] = grow(idx[~left])
        return me

    grow(np.arange(len(x)))
    return cells


def _lists(cells, leaves, theta, r_kern=2.0):
    """Far and near (leaf ordinal, cell) pairs of the leaf-only walk."""
    dev = "cuda"
    com = torch.tensor(np.array([c[1] for c in cells]), device=dev)
    size = torch.tensor([c[2] for c in cells], device=dev, dtype=F64)
    hmax = torch.tensor([float(c[3]) for c in cells], device=dev, dtype=F64)
    left = torch.tensor([c[4] for c in cells], device=dev)
    right = torch.tensor([c[5] for c in cells], device=dev)
    leaf_cell = torch.tensor(leaves, device=dev)
    k, b = torch.arange(len(leaves), device=dev), torch.zeros(len(leaves), device=dev, dtype=torch.long)
    far, near = [], []
    while k.numel():
        a = leaf_cell[k]
        d = com[a] - com[b]
        r2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        reach = (size[a] + size[b]) + r_kern * torch.maximum(hmax[a], hmax[b])
        opened = (r2 == 0) | ((theta * theta) * r2 < size[b] * size[b]) | (r2 < reach * reach)
        opened |= theta == 0.0
        is_leaf = left[b] < 0
        far.append(torch.stack([k[~opened], b[~opened]]))
        near.append(torch.stack([k[opened & is_leaf], b[opened & is_leaf]]))
        down = opened & ~is_leaf
        k, b = torch.cat([k[down], k[down]]), torch.cat([left[b[down]], right[b[down]]])
    return torch.cat(far, 1), torch.cat(near, 1)


def _spline(r, h):
    """Force over distance and potential of the M4-softened unit mass."""
    q = r / h
    inner = 4.0 / 3.0 + q * q * (-1.2 + 0.5 * q)
    outer = 8.0 / 3.0 - 3.0 * q + 1.2 * q ** 2 - q ** 3 / 6.0 - 1.0 / (15.0 * q ** 3)
    f = torch.where(q < 1, inner / h ** 3, torch.where(q < 2, outer / h ** 3, r ** -3))
    inner = 1.4 - 2.0 / 3.0 * q ** 2 + 0.3 * q ** 4 - 0.1 * q ** 5
    outer = 1.6 - 4.0 / 3.0 * q ** 2 + q ** 3 - 0.3 * q ** 4 + q ** 5 / 30.0 - 1.0 / (15.0 * q)
    return f, torch.where(q < 1, inner / h, torch.where(q < 2, outer / h, 1.0 / r))


def _field(x, m, h, eps, cells, leaves, far, near):
    """(a, phi) of the particles from the lists, differentiable in x and m."""
    dev, n, n_cells = "cuda", x.shape[0], len(cells)
    # moments of every cell from its particles: M, com, Q = sum m (3 y y - |y|^2 I)
    rows = torch.tensor(np.concatenate([np.full(len(c[0]), i) for i, c in enumerate(cells)]), device=dev)
    cols = torch.tensor(np.concatenate([c[0] for c in cells]), device=dev)
    M = torch.zeros(n_cells, device=dev, dtype=F64).index_add(0, rows, m[cols])
    com = torch.zeros(n_cells, 3, device=dev, dtype=F64).index_add(0, rows, m[cols, None] * x[cols]) / M[:, None]
    y = x[cols] - com[rows]
    eye = torch.eye(3, device=dev, dtype=F64)
    q = m[cols, None, None] * (3.0 * y[:, :, None] * y[:, None, :] - y.square().sum(1)[:, None, None] * eye)
    Q = torch.zeros(n_cells, 3, 3, device=dev, dtype=F64).index_add(0, rows, q)
    del q, y
    leaf_cell = torch.tensor(leaves, device=dev)
    L = len(leaves)
    C0, C1 = torch.zeros(L, device=dev, dtype=F64), torch.zeros(L, 3, device=dev, dtype=F64)
    C2 = torch.zeros(L, 3, 3, device=dev, dtype=F64)
    C3 = torch.zeros(L, 3, 3, 3, device=dev, dtype=F64)

    def sym(t):                                   # t_a,bc + t_b,ac + t_c,ab
        return t + t.permute(0, 2, 1, 3) + t.permute(0, 3, 2, 1)

    for k, b in zip(far[0].split(1 << 18), far[1].split(1 << 18)):
        R = com[leaf_cell[k]] - com[b]
        r2 = R.square().sum(1)
        g = [r2 ** -0.5]
        for o in range(1, 6):
            g.append(-(2 * o - 1) * g[-1] / r2)
        u = torch.einsum("pij,pj->pi", Q[b], R)
        qs = (R * u).sum(1) / 6.0
        s = [-M[b] * g[o] - g[o + 2] * qs for o in range(4)]
        t = [-g[o] / 3.0 for o in range(5)]
        RR = R[:, :, None] * R[:, None, :]
        Ru = R[:, :, None] * u[:, None, :]
        C0 = C0.index_add(0, k, s[0])
        C1 = C1.index_add(0, k, s[1][:, None] * R + t[2][:, None] * u)
        e = [v[:, None, None] for v in (s[1], s[2], t[2], t[3])]
        C2 = C2.index_add(0, k, e[1] * RR + e[0] * eye + e[3] * (Ru + Ru.transpose(1, 2)) + e[2] * Q[b])
        e = [v[:, None, None, None] for v in (s[2], s[3], t[3], t[4])]
        C3 = C3.index_add(0, k, e[1] * R[:, :, None, None] * RR[:, None] + e[0] * sym(R[:, :, None, None] * eye) +
                          e[3] * sym(u[:, :, None, None] * RR[:, None]) +
                          e[2] * sym(R[:, :, None, None] * Q[b][:, None] + u[:, :, None, None] * eye))
    # the expansions at the leaves' particles
    count = torch.tensor([len(cells[c][0]) for c in leaves], device=dev)
    order = torch.tensor(np.concatenate([cells[c][0] for c in leaves]), device=dev)
    start = torch.cumsum(count, 0) - count
    of = torch.repeat_interleave(torch.arange(L, device=dev), count)
    d = x[order] - com[leaf_cell[of]]
    v = torch.einsum("pij,pj->pi", C2[of], d)
    w = torch.einsum("pijk,pj,pk->pi", C3[of], d, d)
    a = torch.zeros(n, 3, device=dev, dtype=F64).index_add(0, order, -(C1[of] + v + 0.5 * w))
    phi = torch.zeros(n, device=dev, dtype=F64).index_add(
        0, order, C0[of] + (C1[of] * d).sum(1) + 0.5 * (v * d).sum(1) + (w * d).sum(1) / 6.0)
    # direct sums over the near lists
    ordinal = torch.full((n_cells,), -1, device=dev)
    ordinal[leaf_cell] = torch.arange(L, device=dev)
    for k, b in zip(near[0].split(1 << 15), near[1].split(1 << 15)):
        b = ordinal[b]
        size = count[k] * count[b]
        e = torch.repeat_interleave(torch.arange(len(k), device=dev), size)
        at = torch.arange(e.numel(), device=dev) - (torch.cumsum(size, 0) - size)[e]
        i = order[start[k][e] + at // count[b][e]]
        j = order[start[b][e] + at % count[b][e]]
        i, j = i[i != j], j[i != j]
        d = x[i] - x[j]
        r2 = d.square().sum(1)
        if h is None:
            p = (r2 + eps * eps) ** -0.5
            f = p ** 3
        else:
            r = torch.sqrt(r2)
            (fi, pi), (fj, pj) = _spline(r, h[i]), _spline(r, h[j])
            f, p = 0.5 * (fi + fj), 0.5 * (pi + pj)
        a = a.index_add(0, i, -(m[j] * f)[:, None] * d)
        phi = phi.index_add(0, i, -m[j] * p)
    return a, phi


def exact(case, seed):
    if case["do"] not in ("step", "grad") or case["n"] > (40000 if case["do"] == "step" else 20000):
        return None                                # too long in plain torch, or (dual walk, integrator) another method
    s = _inputs(case, seed)
    x, m, h, eps = s["x"], s["m"], s["h"], EPS[case["set"]]
    hn = np.full(case["n"], eps) if h is None else h.cpu().numpy()
    cells = _tree(x.cpu().numpy(), m.cpu().numpy(), hn, case["n_leaf"])
    leaves = [i for i, c in enumerate(cells) if c[4] < 0]
    lists = _lists(cells, leaves, case["theta"])
    if case["do"] == "grad":
        x.requires_grad_(True)
        m.requires_grad_(True)
        a, _ = _field(x, m, h, eps, cells, leaves, *lists)
        x_bar, m_bar = torch.autograd.grad(a, (x, m), s["a_bar"])
        return {"a": a, "x_bar": x_bar, "m_bar": m_bar}
    a, phi = _field(x, m, h, eps, cells, leaves, *lists)
    return {"a": a, "phi": phi, "force": (m[:, None] * a).sum(0)}
