"""Boundary nodes in blocks of their own (levels in the flags-first form)
against the same update with the boundary rows in the colour kernels' own
blocks (levels in the speculative form): one FP32 Uzawa step and the residual
from the same random state.  Both forms evaluate the same expressions per
node, so they differ by contraction of multiply-adds at most: 1e-6 of the
field's maximum (16 units in the last place of FP32)."""
import numpy as np
import pytest

from tests.helpers import macro_by_name, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


@pytest.mark.parametrize("cbz", [1, 4])
@pytest.mark.parametrize("name,level", [("cube", 2), ("cube", 5), ("partial", 3), ("slip_cube", 3),
                                        ("slip_obstacle", 3), ("slip_channel", 2), ("sheared", 3)])
def test_boundary_blocks(pkg, name, level, cbz):
    macro = macro_by_name(name)
    out = []
    for spec in (-1, 0):
        mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=min(2, level - 1),
                        spec_max_nodes=spec, colour_block_z=cbz)
        n = mesh.num_nodes(level)
        rng = np.random.default_rng(3)
        for field in ("U", "F"):
            mesh.level_field(level, field, 1, rng.standard_normal((n, 3)))
        for field in ("P", "G"):
            mesh.level_field(level, field, 1, rng.standard_normal(n))
        mesh.level_op(level, "uzawa_step", 1)
        mesh.level_op(level, "residual", 1)
        out.append([mesh.level_field(level, f, 1) for f in ("U", "P", "RU", "RP")])
        mesh.close()
    for a, b in zip(*out):
        assert np.abs(b).max() > 0 and rel_err(a, b) < 1e-6
