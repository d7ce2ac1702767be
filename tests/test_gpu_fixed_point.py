"""GPU: the float64 stencil sums on the integer pipe (csrc/mg_fixed.cuh).

The neighbours of a cell are summed as integers aligned to their largest exponent; cells
whose neighbours are all tiny, or not finite, are summed in FP64 arithmetic.  Both give the
oracle's solution; scaling the source by a power of two scales every output exactly as
long as the same route is taken.
"""

import numpy as np
import pytest

from oracle.multigrid import solve as oracle_solve
from synthetic import Geometry, NestSpec, make_delta

pytestmark = pytest.mark.gpu
# both sides run the same V-cycles: only rounding differs (order 1e-15 per operation, a few
# hundred operations deep), and the oracle tests of this repository allow 1e-10
TOL = 1e-10

GEOMS = {
    2: Geometry((20, 36, 34), 10.0, 2, (NestSpec((18, 22, 26), (5, 9, 11)),)),
    4: Geometry((24, 20, 44), 10.0, 4, (NestSpec((20, 12, 38), (6, 7, 13)),)),
    6: Geometry((28, 40, 36), 10.0, 6, (NestSpec((16, 34, 22), (9, 11, 12)),)),
}


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_6031_gb300 as pkg
    return pkg


def solve(lib, geom, deltas):
    import torch
    h = lib.Hierarchy(lib.config_from_geometry(geom, tol=0.0, max_cycles=3))
    phis, _ = h.solve_1lpt([torch.from_numpy(np.ascontiguousarray(d)).cuda() for d in deltas],
                           allow_noconv=True)
    out = [p.cpu().numpy() for p in phis]
    h.close()
    return out


def source(geom, kind):
    deltas = make_delta(geom, 5)
    if kind == "spikes":
        # one cell in some thousand carries nearly everything, the rest is 12 orders below
        rng = np.random.Generator(np.random.PCG64(9))
        deltas = [1e-12 * d + (rng.random(d.shape) < 1e-3) * rng.standard_normal(d.shape)
                  for d in deltas]
    return deltas


@pytest.mark.parametrize("kind", ["field", "spikes"])
@pytest.mark.parametrize("order", (2, 4, 6))
def test_scaled_sources(lib, order, kind):
    geom = GEOMS[order]
    deltas = source(geom, kind)
    ref, _ = oracle_solve(geom, deltas, tol=0.0, cycles=3)
    plain = solve(lib, geom, deltas)
    for a, b in zip(plain, ref):
        assert np.sqrt(np.sum((a - b) ** 2) / np.sum(b * b)) < TOL
    for k in (200, -200):  # the integer route: exact scaling
        for a, b in zip(solve(lib, geom, [np.ldexp(d, k) for d in deltas]), plain):
            assert np.array_equal(a, np.ldexp(b, k)), k
    # potentials below 2^-926: the FP64 route
    for a, b in zip(solve(lib, geom, [np.ldexp(d, -940) for d in deltas]), ref):
        a = np.ldexp(a, 940)
        assert np.sqrt(np.sum((a - b) ** 2) / np.sum(b * b)) < TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_source_that_is_not_finite(lib, bad):
    geom = GEOMS[6]
    deltas = source(geom, "field")
    deltas[0][3, 5, 7] = bad
    assert all(np.isnan(p).any() for p in solve(lib, geom, deltas))
