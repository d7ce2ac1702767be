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


# levels of at least 2^17 cells are worked on in tiles of 8 x 8 x 32 cells: sides with
# remainders along every axis, a nest whose faces cut tiles
TILED = {
    2: Geometry((60, 44, 52), 10.0, 2, (NestSpec((58, 50, 46), (10, 8, 9)),)),
    4: Geometry((52, 44, 60), 10.0, 4, (NestSpec((46, 42, 70), (9, 7, 11)),)),
    6: Geometry((44, 60, 52), 10.0, 6, (NestSpec((50, 66, 42), (8, 12, 11)),)),
}


@pytest.mark.parametrize("order", (2, 4, 6))
def test_tiled_levels(lib, order):
    """One whole step (solves, tau, displacements) against the oracle at matched cycles."""
    import torch
    from oracle.lpt import lpt_pipeline
    geom = TILED[order]
    deltas = make_delta(geom, 7)
    ref = lpt_pipeline(geom, deltas, tol=0.0, cycles=2)
    h = lib.Hierarchy(lib.config_from_geometry(geom, tol=0.0, max_cycles=2))
    out, i1, i2 = h.pipeline([torch.from_numpy(np.ascontiguousarray(d)).cuda() for d in deltas])
    np.testing.assert_allclose(i1["history"], ref["info1"]["history"], rtol=1e-6, atol=1e-14)
    np.testing.assert_allclose(i2["level_rel_residual"], ref["info2"]["level_rel_residual"],
                               rtol=1e-6, atol=1e-14)

    def off(a, b):
        a = a.cpu().numpy()
        return np.sqrt(np.sum((a - b) ** 2) / np.sum(b * b))

    for l in range(2):
        assert off(out["phi1"][l], ref["phi1"][l]) < TOL
        assert off(out["phi2"][l], ref["phi2"][l]) < TOL
        for a in range(3):
            assert off(out["disp1"][3 * l + a], ref["psi1"][l][a]) < TOL
            assert off(out["disp2"][3 * l + a], ref["psi2"][l][a]) < TOL
    # the same source 2^-940 times smaller takes the FP64 route in every tile
    tiny, _, _ = h.pipeline([torch.from_numpy(np.ldexp(d, -940)).cuda() for d in deltas],
                            allow_noconv=True)
    for l in range(2):
        assert off(torch.ldexp(tiny["phi1"][l], torch.tensor(940.0, dtype=torch.float64,
                                                             device="cuda")),
                   ref["phi1"][l]) < TOL
    h.close()


@pytest.mark.parametrize("shape", [(4, 4, 4), (20, 36, 34), (12, 8, 70), (20, 24, 35), (3, 5, 6)])
@pytest.mark.parametrize("order", (2, 4, 6))
def test_tau_of_one_periodic_level(lib, order, shape):
    """tau of a single periodic level is read and written dense where its rows are even, phi
    is 16-byte aligned and the arrays are apart, and through padded copies otherwise; both
    match the oracle, also where every tile takes the FP64 route."""
    import torch
    from oracle.hierarchy import Hierarchy as OracleHierarchy
    from oracle.lpt import lpt2_source as oracle_tau
    geom = Geometry(shape, 7.0, order, ())
    x = np.random.Generator(np.random.PCG64(2)).standard_normal(shape)
    want = oracle_tau(OracleHierarchy(geom), [x])[0]
    h = lib.Hierarchy(lib.config_from_geometry(geom))

    def off(a, b):
        a = a.cpu().numpy()
        return np.sqrt(np.sum((a - b) ** 2) / np.sum(b * b))

    phi = torch.from_numpy(x).cuda()
    assert off(h.lpt2_source([phi])[0], want) < TOL
    shifted = torch.empty(phi.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(shape)
    shifted.copy_(phi)
    assert off(h.lpt2_source([shifted])[0], want) < TOL
    tiny = torch.from_numpy(np.ldexp(x, -480)).cuda()
    assert off(torch.ldexp(h.lpt2_source([tiny])[0],
                           torch.tensor(960.0, dtype=torch.float64, device="cuda")), want) < TOL
    # in place
    from paper_1103_6031_gb300.mg import _ptrs
    assert h.lib.mg_lpt2_source(h.h, _ptrs([phi]), _ptrs([phi])) == 0
    assert off(phi, want) < TOL
    h.close()


@pytest.mark.parametrize("shape", [(4, 4, 4), (20, 36, 34), (12, 8, 70), (20, 24, 35), (3, 5, 6)])
@pytest.mark.parametrize("order", (2, 4, 6))
def test_local_density_of_one_periodic_level(lib, order, shape):
    """The local density of a single periodic level goes through dense arrays where its rows
    are even and through padded ones otherwise; both match the oracle, with an output that is
    one of the inputs or starts on an odd element too."""
    import torch
    from oracle.hierarchy import Hierarchy as OracleHierarchy
    from oracle.lpt import lla_density as oracle_lla
    from paper_1103_6031_gb300.mg import _ptrs
    geom = Geometry(shape, 7.0, order, ())
    rng = np.random.Generator(np.random.PCG64(4))
    x, y = rng.standard_normal(shape), rng.standard_normal(shape)
    # second derivatives of 0.1 at most: no shell crossing
    hh = (7.0 / shape[0]) ** 2
    a1, a2 = 0.1 * hh / (40 * np.abs(x).max()), 0.04 * hh / (40 * np.abs(y).max())
    want = oracle_lla(OracleHierarchy(geom), [x], [y], a1, a2)[0]
    h = lib.Hierarchy(lib.config_from_geometry(geom))

    def off(a):
        a = a.cpu().numpy()
        return np.sqrt(np.sum((a - want) ** 2) / np.sum((want - 1.0) ** 2))

    p, q = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    # rho - 1 is about 1e-3, stored next to 1 (2^-53)
    assert off(h.lla_density([p], [q], a1, a2)[0]) < TOL
    odd = torch.empty(p.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(shape)
    for out in (odd, p):
        assert h.lib.mg_lla_density(h.h, _ptrs([p]), _ptrs([q]), a1, a2, _ptrs([out])) == 0
        assert off(out) < TOL
    h.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_source_that_is_not_finite(lib, bad):
    geom = GEOMS[6]
    deltas = source(geom, "field")
    deltas[0][3, 5, 7] = bad
    assert all(np.isnan(p).any() for p in solve(lib, geom, deltas))
