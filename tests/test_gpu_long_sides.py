"""GPU: the Fourier parts on a nest whose zero-padded side passes 65535 cells, the limit of a
launch grid's second and third dimension (nests are up to twice their parent long, so a side of
33000 lies four levels below the largest base)."""

import numpy as np
import pytest

from synthetic import Geometry, NestSpec, PowerLaw

pytestmark = pytest.mark.gpu

LONG = (4096, 8176, 16336, 32656, 33000)


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_6031_gb300 as pkg
    return pkg


def geometry(axis):
    """Base and nests that are long along one axis, 16 and 8 cells along the others."""
    def along(a, long, short):
        return tuple(long if b == a else short for b in range(3))
    nests = tuple(NestSpec(along(axis, n, 8), along(axis, 4, 6 if l == 0 else 2))
                  for l, n in enumerate(LONG[1:]))
    return Geometry(along(axis, LONG[0], 16), 4096.0, 2, nests)


def correction(f, h):
    """The isolated order-2 correction i h [t_j / t^2 - sin t_j / lam] f, lam = sum 4 sin^2(t/2),
    with the differences of the two fractions formed axis by axis in extended precision (in
    double, as the oracle forms them, they cancel: eps / t^3 at the smallest t = 2 pi / 66000)."""
    N = [2 * n for n in f.shape]
    t, lam, dlam, dgam = [], [], [], []
    for a, n in enumerate(N):
        i = np.arange(n if a < 2 else n // 2 + 1)
        x = 2 * np.arccos(np.longdouble(-1)) * np.where(i <= n // 2, i, i - n) / n
        shape = [-1 if b == a else 1 for b in range(3)]
        for out, v in ((t, x), (lam, 4 * np.sin(x / 2) ** 2), (dlam, 4 * np.sin(x / 2) ** 2 - x * x),
                       (dgam, np.sin(x) - x)):
            out.append(v.astype(float).reshape(shape))
    t2 = sum(v * v for v in t)
    den = t2 * sum(lam)
    den[0, 0, 0] = 1.0
    F = np.fft.rfftn(f, s=N, axes=(0, 1, 2))
    out = []
    for a in range(3):
        c = h * (t[a] * sum(dlam) - dgam[a] * t2) / den
        c = np.where(np.abs(t[a]) > 3.14159, 0.0, c)  # the Nyquist plane
        out.append(np.fft.irfftn(1j * c * F, s=N, axes=(0, 1, 2))[tuple(slice(0, n) for n in f.shape)])
    return out


@pytest.mark.parametrize("axis", (0, 1))
def test_hybrid(lib, axis):
    import torch
    geom = geometry(axis)
    shape = geom.nests[-1].n
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    f = np.random.Generator(np.random.PCG64(3)).standard_normal(shape)
    psi = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(3)]
    h.hybrid_correction(torch.from_numpy(f).cuda(), psi)
    h.close()
    cell = 4096.0 / geom.base_n[0] / 16
    for a, b in zip(psi, correction(f, cell)):
        assert np.sqrt(np.sum((a.cpu().numpy() - b) ** 2) / np.sum(b ** 2)) < 1e-7


@pytest.mark.parametrize("axis", (0, 1))
def test_multiscale_density(lib, axis):
    from oracle.density import multiscale
    geom = geometry(axis)
    dk = 0.01
    k = np.arange(6000) * dk
    table = np.sqrt(PowerLaw(-2.0)(np.maximum(k, 1e-12)))
    table[0] = 0.0
    got = lib.mg.density_multiscale(lib.config_from_geometry(geom), 5, table, dk)
    for g, w in zip(got, multiscale(geom, 5, table, dk)):
        # transforms of up to 2^25 points, each 1e-16 log2 of them
        assert np.sqrt(np.sum((g.cpu().numpy() - w) ** 2) / np.sum(w * w)) < 1e-11
