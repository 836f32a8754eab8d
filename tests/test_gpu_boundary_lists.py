"""Device memory of the boundary lists: a sheared cube, where every node is a
boundary node and none is kept apart, holds one list of its nodes (8 bytes
each) more than the cube of the same lattice, besides its class tables."""
import pytest

from tests.helpers import macro_by_name

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


def test_lists_of_lattices_without_blocks_of_boundary_nodes(pkg):
    level, bytes_ = 6, []
    for name in ("cube", "sheared"):
        macro = macro_by_name(name)
        mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level)
        nodes = sum(mesh.num_nodes(l) for l in range(mesh.coarsest, level + 1))
        bytes_.append(mesh.device_bytes())
        mesh.close()
    tables = 1 << 20
    assert bytes_[1] - bytes_[0] < 8 * nodes + tables
