"""GPU: fields of a wide range inside one tile of the integer stencils (csrc/mg_tile.cuh).

tau, the local density and the displacements of every cell are compared with extended
precision, each cell's error against the values in its own stencil: a strong cell must not
take bits from the weak cells that share its tile but not their stencils.
"""

import numpy as np
import pytest

from synthetic import Geometry, NestSpec

pytestmark = pytest.mark.gpu

LD = np.longdouble
LAP = {2: (-2, 1), 4: (-30, 16, -1), 6: (-490, 270, -27, 2)}
LAP_DEN = {2: 1, 4: 12, 6: 180}
GRAD = {2: (1,), 4: (8, -1), 6: (45, -9, 1)}
GRAD_DEN = {2: 2, 4: 12, 6: 60}
EPS = 2.0 ** -53
# h^2 phi'' and h phi' relative to the largest value in the stencil.  In FP64 the weights add
# up to 6.1 at most and meet 5 roundings; as integers at most 22 units (a mixed derivative's) of
# 2^-52 of that value.
D_EPS = 48 * EPS
# remainders along every axis; 2^17 cells, where displacements are formed on tiles, and odd rows,
# which are read padded
SHAPES = [(52, 44, 60), (26, 28, 35)]


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_6031_gb300 as pkg
    return pkg


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def roll(u, s, a):
    return np.roll(u, -s, a)


def second(u, a, order):
    w = LAP[order]
    return sum((LD(w[s]) * (roll(u, s, a) + roll(u, -s, a)) for s in range(1, len(w))),
               LD(w[0]) * u) / LD(LAP_DEN[order])


def first(u, a, order):
    return sum(LD(w) * (roll(u, s, a) - roll(u, -s, a))
               for s, w in enumerate(GRAD[order], 1)) / LD(GRAD_DEN[order])


def reach(u, axes, order):
    """The largest magnitude within order / 2 cells along the axes (all combinations)."""
    m = np.abs(u)
    for a in axes:
        m = np.max([roll(m, s, a) for s in range(-(order // 2), order // 2 + 1)], axis=0)
    return m


def hessian(phi, order):
    """d, m and the largest value in the Hessian's stencil, h = 1."""
    u = phi.astype(LD)
    d = [second(u, a, order) for a in range(3)]
    m = [first(first(u, b, order), a, order) for a, b in ((0, 1), (0, 2), (1, 2))]
    q = np.max([reach(phi, ab, order) for ab in ((0, 1), (0, 2), (1, 2))], axis=0)
    return d, m, q


def tau_and_bound(phi, order):
    d, m, q = hessian(phi, order)
    pairs = ((0, 1), (0, 2), (1, 2))
    tau = sum(d[a] * d[b] for a, b in pairs) - sum(v * v for v in m)
    e = D_EPS * q
    bound = sum(2 * e * np.abs(v) + e * e for v in d + m) + \
        16 * EPS * (sum(np.abs(d[a] * d[b]) for a, b in pairs) + sum(v * v for v in m))
    return tau, bound


def field(kind, shape):
    rng = np.random.Generator(np.random.PCG64(11))
    x = rng.standard_normal(shape)
    r2 = sum(((np.arange(n) - (0.4 * n + 0.2)) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
             for a, n in enumerate(shape))
    if kind == "gauss":  # 2 cells wide
        return np.exp(-r2 / 8.0)
    if kind == "spike":  # one cell 2^60 above the rest, another 2^30
        x[17, 19, 20] = 2.0 ** 60
        x[11, 6, 33] = -2.0 ** 30
        return x
    if kind == "half":   # nothing on one side, deep below the other's values on a plane
        x[:, : shape[1] // 2] = 0.0
        x[:, shape[1] // 2 + 7] *= 2.0 ** -70
        return x
    return np.ldexp(x, -60 * (r2 > 150))  # island: a ball of ordinary values in tiny ones


KINDS = ["gauss", "spike", "half", "island"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", (2, 4, 6))
def test_one_level(lib, order, shape, kind):
    geom = Geometry(shape, float(shape[0]), order, ())  # h = 1
    phi = field(kind, shape)
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    tau, bound = tau_and_bound(phi, order)
    off = np.abs(h.lpt2_source([dev(phi)])[0].cpu().numpy() - tau)
    assert np.all(off <= bound), float(np.max(off[off > bound] / bound[off > bound]))
    psi = h.displacements([dev(phi)])[0]
    tol = 24 * EPS * reach(phi, (0,), order)
    for a in (1, 2):
        tol = np.maximum(tol, 24 * EPS * reach(phi, (a,), order))
    for a in range(3):
        off = np.abs(psi[a].cpu().numpy() + first(phi.astype(LD), a, order))
        assert np.all(off <= tol), a
    h.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", (2, 4, 6))
def test_local_density(lib, order, shape):
    """Weak cells whose second derivatives are a few per cent beside one of 2^60."""
    geom = Geometry(shape, float(shape[0]), order, ())
    phi = field("spike", shape)
    phi[11, 6, 33] = 1.0
    a1 = 2.0 ** -9
    d, m, q = hessian(phi, order)
    a, b, c = (1 - LD(a1) * v for v in d)
    m = [LD(a1) * v for v in m]
    rho = 1 / (a * b * c - a * m[2] ** 2 - b * m[1] ** 2 - c * m[0] ** 2 - 2 * m[0] * m[1] * m[2])
    rho = rho - rho.mean() + 1
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    off = np.abs(h.lla_density([dev(phi)], a1=a1)[0].cpu().numpy() - rho)
    weak = q < 2.0 ** 20
    # 1 / det is of order 1 there, off by the Hessian's 48 EPS a1 q a few times over and some ten
    # roundings; the mean of 10^5 cells adds its own
    assert off[weak].max() < 1e-13
    h.close()


@pytest.mark.parametrize("order", (2, 4, 6))
def test_nest(lib, order):
    """Strong cells inside a nest and beside its face, in tiles that the face cuts."""
    n0, n1, off = (44, 60, 52), (50, 66, 42), (8, 12, 11)
    geom = Geometry(n0, float(n0[0]), order, (NestSpec(n1, off),))
    base = np.random.Generator(np.random.PCG64(12)).standard_normal(n0)
    box = tuple(slice(o, o + s // 2) for o, s in zip(off, n1))
    nest = base[box].repeat(2, 0).repeat(2, 1).repeat(2, 2)  # covered cells: their exact means
    nest[8:10, 30:32, 8:10] = 2.0 ** 60
    base[box][4, 15, 4] = 2.0 ** 60
    base[6, 20, 30] = -2.0 ** 50  # two cells outside the nest's low x face
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    got = h.lpt2_source([dev(base), dev(nest)])
    for l, (phi, keep) in enumerate(((base, np.ones(n0, bool)), (nest, np.zeros(n1, bool)))):
        if l == 0:
            keep[box] = False  # the mean of the children
        else:
            keep[3:-3, 3:-3, 3:-3] = True  # no interpolated ghosts in the stencils
        tau, bound = tau_and_bound(phi, order)
        s = 16.0 ** l  # h = 1/2 on the nest
        err = np.abs(got[l].cpu().numpy() - s * tau)
        assert np.all(err[keep] <= s * bound[keep]), l
    psi = h.displacements([dev(base), dev(nest)])
    for l, phi in enumerate((base, nest)):
        keep = np.ones(phi.shape, bool)
        if l:
            keep[:] = False
            keep[3:-3, 3:-3, 3:-3] = True
        tol = 24 * EPS * np.max([reach(phi, (a,), order) for a in range(3)], axis=0) * 2 ** l
        for a in range(3):
            err = np.abs(psi[l][a].cpu().numpy() + 2 ** l * first(phi.astype(LD), a, order))
            assert np.all(err[keep] <= tol[keep]), (l, a)
    h.close()
