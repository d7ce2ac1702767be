"""GPU: mixed derivatives on fields that alternate at the grid scale.

The signs are those for which the antisymmetric weights of order 6, applied along one axis
to their own result along another, add up with nothing cancelling, every value close below a
power of two: the largest sums the integer stencils can meet.
"""

import numpy as np
import pytest

from oracle.hierarchy import Hierarchy as OracleHierarchy
from oracle.lpt import lla_density as oracle_lla
from oracle.lpt import lpt2_source as oracle_tau
from synthetic import Geometry, NestSpec

pytestmark = pytest.mark.gpu

# signs at offsets 0, 1, .. 7 (7 = -1): odd about 0
OUTER = (1, -1, -1, 1, 1, -1, 1, 1)
INNER = (1, 1, -1, 1, 1, -1, 1, -1)
PAIRS = [(0, 1), (0, 2), (1, 2)]
# |phi| <= 2, h = 1: entries of the Hessian reach 2 * 6.1, tau 3 * 12.2^2 = 450, summed in some
# 50 roundings of 1.1e-16
TAU_TOL = 450 * 50 * 1.2e-16
# Hessian / 2^7: entries below 0.1, 1 / det below 1.6, some 100 roundings of 2e-16
LLA_TOL = 4e-14


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_6031_gb300 as pkg
    return pkg


def pattern(shape, pair, a):
    f = np.full(shape, a)
    for axis, signs in zip(pair, (OUTER, INNER)):
        s = np.resize(np.array(signs, float), shape[axis])
        f *= s.reshape([-1 if q == axis else 1 for q in range(3)])
    return f


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


# even rows: dense route; odd rows: padded route
@pytest.mark.parametrize("shape", [(16, 24, 40), (24, 16, 43)])
@pytest.mark.parametrize("pair", PAIRS)
@pytest.mark.parametrize("order", (2, 4, 6))
def test_one_level(lib, order, pair, shape):
    geom = Geometry(shape, float(shape[0]), order, ())
    x = pattern(shape, pair, 1.99)
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    tau = h.lpt2_source([dev(x)])[0].cpu().numpy()
    assert np.abs(tau - oracle_tau(OracleHierarchy(geom), [x])[0]).max() < TAU_TOL
    rho = h.lla_density([dev(x)], a1=2.0 ** -7)[0].cpu().numpy()
    assert np.abs(rho - oracle_lla(OracleHierarchy(geom), [x], a1=2.0 ** -7)[0]).max() < LLA_TOL
    h.close()


@pytest.mark.parametrize("pair", PAIRS)
def test_nest(lib, pair):
    geom = Geometry((24, 32, 40), 24.0, 6, (NestSpec((16, 24, 32), (7, 9, 8)),))
    x = [pattern(n, pair, 1.99) for n in ((24, 32, 40), (16, 24, 32))]
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    got = h.lpt2_source([dev(v) for v in x])
    want = oracle_tau(OracleHierarchy(geom), x)
    off = [np.abs(g.cpu().numpy() - w) for g, w in zip(got, want)]
    off[0][7:15, 9:21, 8:24] = 0.0  # covered: the mean of the children
    assert off[0].max() < TAU_TOL
    # cells of the nest whose stencils hold no interpolated ghosts; h = 1/2
    assert off[1][3:-3, 3:-3, 3:-3].max() < 16 * TAU_TOL
    h.close()
