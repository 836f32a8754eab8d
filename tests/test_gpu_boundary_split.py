"""Boundary nodes in blocks of their own on levels that have them: a level is
split where fewer than half of its pressure nodes are boundary nodes (in FP32
only in the flags-first form).  One Uzawa step and the residual in both
precisions, both node forms and both operator forms against the oracle: FP64
1e-11 and FP32 1e-5 per step, ten times that for the residual of the result, as
in the tests of the slip and D-form smoothers."""
import numpy as np
import pytest

from oracle import multigrid as MG
from tests.helpers import macro_by_name, p_from_lattice, p_to_lattice, rel_err, u_from_lattice, u_to_lattice

pytestmark = pytest.mark.gpu

MESHES = [("cube", 4), ("partial", 4), ("slip_cube", 4), ("slip_obstacle", 3), ("channel", 2)]
_oracle = {}


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


def _expected(name, level, form):
    """Random admissible state, the oracle's state after one step, and its residual."""
    if (name, level, form) not in _oracle:
        H = MG.build_hierarchy(macro_by_name(name), level, coarsest=level - 1, form="D" if form else "laplace")
        L, rng = H.levels[level], np.random.default_rng(31)
        g = rng.standard_normal(L.n_p)
        if L.pure_dirichlet:
            g -= g.mean()
        st = (L.proj(rng.standard_normal((3, L.n_u))), rng.standard_normal(L.n_p),
              L.proj(rng.standard_normal((3, L.n_u))), g)
        u, p, f, g = (a.copy() for a in st)
        MG.uzawa_step(H, level, u, p, f, g)
        _oracle[name, level, form] = (L, st, (u, p), L.residual(u, p, f, g))
    return _oracle[name, level, form]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spec,cbz", [(-1, 1), (-1, 4), (0, 1)])
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("name,level", MESHES)
def test_split_levels(pkg, name, level, form, spec, cbz, precision):
    macro = macro_by_name(name)
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=level - 1, operator_form=form,
                    spec_max_nodes=spec, colour_block_z=cbz)
    fl = mesh.node_flags()
    assert 0 < 2 * np.count_nonzero(fl & 4) < np.count_nonzero(fl & 1)
    L, (u, p, f, g), (ou, op), (oru, orp) = _expected(name, level, form)
    dims, tol = mesh.dims(), (1e-5 if precision else 1e-11)
    for field, v in (("U", u_to_lattice(L, dims, u)), ("P", p_to_lattice(L, dims, p)), ("F", u_to_lattice(L, dims, f)),
                     ("G", p_to_lattice(L, dims, g))):
        mesh.level_field(level, field, precision, v)
    mesh.level_op(level, "uzawa_step", precision)
    assert rel_err(u_from_lattice(L, dims, mesh.level_field(level, "U", precision)), ou) < tol
    assert rel_err(p_from_lattice(L, dims, mesh.level_field(level, "P", precision)), op) < tol
    mesh.level_op(level, "residual", precision)
    assert rel_err(u_from_lattice(L, dims, mesh.level_field(level, "RU", precision)), oru) < 10 * tol
    assert rel_err(p_from_lattice(L, dims, mesh.level_field(level, "RP", precision)), orp) < 10 * tol
    mesh.close()
