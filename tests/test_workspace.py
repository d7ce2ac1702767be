"""Device bytes a hierarchy takes (mg_workspace_bytes), against the arrays its calls use (CPU)."""

import paper_1103_6031_gb300 as pkg


def padded(n, g):
    return (n + 2 * g) ** 2 * ((4 + n + g + 7) // 8 * 8) * 8


def test_one_periodic_level():
    n, g = 128, 3
    got = pkg.workspace_bytes(pkg.make_config((n, n, n), 1.0, 2 * g, []))
    sides = [128, 64, 32, 16, 8]
    # u twice and the source of every level, the leaf's own source; dense: Phi of the local
    # density and the staged phi and displacements
    need = sum(3 * padded(s, g) for s in sides) + padded(n, g) + 5 * 8 * n ** 3
    # ubar of the coarse levels, partial sums, the coarsest level's table, alignment
    assert need < got < need + 8 * n ** 3 // 7 + 100000


def test_hybrid():
    n = (34, 18, 26)
    base, nests = (40, 28, 36), [(n, (9, 8, 10))]
    plain = pkg.workspace_bytes(pkg.make_config(base, 1.0, 6, nests))
    hybrid = pkg.workspace_bytes(pkg.make_config(base, 1.0, 6, nests, hybrid=True))
    spectrum = 16 * 68 * 36 * 27
    # a copy of the source, the level's planes of the padded grid, two half spectra and one of
    # work area, small tables
    need = 8 * 34 * 18 * 26 + 8 * 34 * 36 * 52 + 3 * spectrum
    assert need <= hybrid - plain < need + 10000
