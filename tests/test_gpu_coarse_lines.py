"""The coarse solve on both sides of the lines between its shapes: one thread
block and the cluster (320 velocity rows, 256 coupled rows, 4,096 unknowns),
one row per lane and vectors in memory (2,560 velocity rows on 16 CTAs), and
row counts that are no multiple of 32.  Against the oracle's coarse solve on a
random state to 1e-9, as in the test over its shapes: the Krylov recurrence
amplifies the rounding-order differences of its sums."""
import numpy as np
import pytest

import workloads as W
from oracle import multigrid as MG
from tests.helpers import p_from_lattice, p_to_lattice, rel_err, u_from_lattice, u_to_lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


# (cells, level, form, slip sides, free velocity nodes or None): without slip prod(cells 2^level - 1)
LINES = [
    ((5, 4, 3), 1, 0, (), 315),      # scalar, one block
    ((7, 4, 2), 1, 0, (), 273),
    ((6, 4, 3), 1, 0, (), 385),      # cluster
    ((1, 1, 1), 3, 0, (), 343),
    ((2, 5, 5), 2, 0, (), 2527),     # a row per lane
    ((2, 4, 7), 2, 0, (), 2835),     # vectors in memory
    ((2, 6, 2), 1, 1, (), 99),       # coupled: 297 rows, cluster
    ((3, 3, 2), 1, 1, (), 75),       # 225, one block
    ((3, 2, 3), 1, 0, ("z0",), None),
    ((4, 3, 3), 1, 0, ("z0", "z1"), None),
    ((2, 2, 1), 3, 1, (), 1575),     # 4,725 coupled rows, more than 4,096 unknowns
    ((4, 4, 4), 1, 1, (), 343),
]


@pytest.mark.parametrize("cells,level,form,slip,rows", LINES)
def test_coarse_solve_lines(pkg, cells, level, form, slip, rows):
    macro = W.box_of_cubes(*cells, slip_sides=slip)
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=level, operator_form=form)
    H = MG.build_hierarchy(macro, level, coarsest=level, form="D" if form else "laplace")
    L, dims = H.levels[level], mesh.dims(level)
    assert rows is None or L.n_u == rows
    rng = np.random.default_rng(12)
    u, p = np.zeros((3, L.n_u)), np.zeros(L.n_p)
    f, g = L.proj(rng.standard_normal((3, L.n_u))), rng.standard_normal(L.n_p)
    g -= g.mean()
    for name, val in (("U", u_to_lattice(L, dims, u)), ("P", p_to_lattice(L, dims, p)),
                      ("F", u_to_lattice(L, dims, f)), ("G", p_to_lattice(L, dims, g))):
        mesh.level_field(level, name, 0, val)
    mesh.level_op(level, "coarse_solve")
    MG.vcycle(H, level, u, p, f, g)  # on the coarsest level: the MINRES correction
    gu = u_from_lattice(L, dims, mesh.level_field(level, "U"))
    gp = p_from_lattice(L, dims, mesh.level_field(level, "P"))
    assert rel_err(gu, u) < 1e-9
    assert rel_err(L.project_pressure(gp), L.project_pressure(p)) < 1e-9
    mesh.close()
