"""The coarse solve over the sizes at which its CG changes shape: one warp per
velocity block with one, two or four rows per lane, one row per thread over a
block or a cluster, vectors in global memory beyond that, for the scalar and
the coupled (D form, free slip) velocity block.  Against the oracle's coarse
solve on a random state to 1e-9: the Krylov recurrence amplifies the
rounding-order differences of its sums, and 1e-9 is far below the 5e-3
tolerance the solver is asked for."""
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


# (cells, level, form, slip sides): free velocity nodes, prod(cells 2^level - 1) without slip
SHAPES = [
    ((1, 1, 1), 0, 0, ()),          # none: pressure unknowns only
    ((2, 1, 1), 0, 1, ()),
    ((1, 1, 1), 1, 0, ()),          # 1
    ((1, 1, 1), 2, 0, ()),          # 27: one row per lane
    ((2, 1, 1), 2, 0, ()),          # 63: two
    ((3, 1, 1), 2, 0, ()),          # 99: four
    ((4, 1, 1), 2, 0, ()),          # 135: cluster
    ((1, 1, 1), 3, 0, ()),          # 343
    ((2, 2, 1), 3, 0, ()),          # 1,575
    ((1, 1, 1), 4, 0, ()),          # 3,375: vectors in memory
    ((1, 1, 1), 2, 1, ()),          # 81 coupled rows, one block
    ((3, 1, 1), 2, 1, ()),          # 297
    ((1, 1, 1), 3, 1, ()),          # 1,029, cluster
    ((2, 1, 1), 3, 0, ("z0",)),     # free slip couples the components
    ((1, 1, 1), 4, 1, ()),          # 10,125: vectors in memory
]


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("cells,level,form,slip", SHAPES)
def test_coarse_solve_shapes(pkg, cells, level, form, slip, zero):
    macro = W.box_of_cubes(*cells, slip_sides=slip)
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=level, operator_form=form)
    H = MG.build_hierarchy(macro, level, coarsest=level, form="D" if form else "laplace")
    L, dims = H.levels[level], mesh.dims(level)
    rng = np.random.default_rng(11)
    u, p = np.zeros((3, L.n_u)), np.zeros(L.n_p)
    f, g = L.proj(rng.standard_normal((3, L.n_u))), rng.standard_normal(L.n_p)
    if zero:
        # one component's first CG has a zero right-hand side and must not run
        f[0] = 0.0
        f, g = L.proj(f), np.zeros(L.n_p)
    g -= g.mean()
    for name, val in (("U", u_to_lattice(L, dims, u)), ("P", p_to_lattice(L, dims, p)),
                      ("F", u_to_lattice(L, dims, f)), ("G", p_to_lattice(L, dims, g))):
        mesh.level_field(level, name, 0, val)
    mesh.level_op(level, "coarse_solve")
    MG.vcycle(H, level, u, p, f, g)  # on the coarsest level: the MINRES correction
    gu = u_from_lattice(L, dims, mesh.level_field(level, "U"))
    gp = p_from_lattice(L, dims, mesh.level_field(level, "P"))
    assert L.n_u == 0 or rel_err(gu, u) < 1e-9
    assert rel_err(L.project_pressure(gp), L.project_pressure(p)) < 1e-9
    mesh.close()
