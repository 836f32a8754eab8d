"""A lattice of 64,001 planes: the grids of the colour and residual kernels
have one block per plane and at most 65,535 along that axis, so the blocks of
their boundary nodes find no room beside them.  One Uzawa step and the
residual of a state that is zero above two cubes equal, in their first three
cubes, those of a short column: the same kernels' arithmetic per node, so they
differ by contraction of multiply-adds at most (1e-13 of the field's maximum in
FP64, 1e-5 in FP32)."""
import numpy as np
import pytest

import workloads as W
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

LEVEL, LONG, SHORT = 4, 4000, 8


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


@pytest.fixture(scope="module")
def meshes(pkg):
    out = []
    for n in (LONG, SHORT):
        macro = W.box_of_cubes(1, 1, n)
        out.append(pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, LEVEL, coarsest_level=LEVEL - 4))
    yield out
    for m in out:
        m.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_long_lattice(meshes, precision):
    plane = 17 * 17
    got = []
    for mesh in meshes:
        n, rng = mesh.num_nodes(), np.random.default_rng(8)
        for field, nc in (("U", 3), ("F", 3), ("P", 1), ("G", 1)):
            x = np.zeros((n, nc))
            x[:33 * plane] = rng.standard_normal((33 * plane, nc))
            mesh.level_field(LEVEL, field, precision, x if nc == 3 else x[:, 0].copy())
        mesh.level_op(LEVEL, "uzawa_step", precision)
        mesh.level_op(LEVEL, "residual", precision)
        got.append([mesh.level_field(LEVEL, f, precision)[:49 * plane] for f in ("U", "P", "RU", "RP")])
    for a, b in zip(*got):
        assert np.abs(b).max() > 0 and rel_err(a, b) < (1e-5 if precision else 1e-13)
