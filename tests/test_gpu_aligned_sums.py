"""FP64 stencil sums where large neighbours cancel and at the ends of the
integers' range: the smoother's and the residual's rows at regular nodes
against the closed forms in extended precision.

Every stencil forms sums of pairs first: differences of opposite neighbours in
the divergences, sums of opposite neighbours in the Laplacian.  A pair of equal
or close values cancels without a rounding error in FP64, so the small values
beside it count in full.  Tolerance: 16 u of the sum over the pairs of
|weight| |pair| (u = 2^-53): the FP64 operations round each pair once, then at
most nine sums of them, and the row's scale factors carry a few u.

"pairs" has large equal opposite neighbours beside small values; "turns" large
values of opposite sign; "extreme" is a checkerboard of the largest mantissas,
which reaches the largest integer sums; "wide" mixes 30 decades; "tiny" and
"huge" lie outside the integers' range."""
import numpy as np
import pytest

from tests.helpers import macro_by_name

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
KUHN = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, 1, 1)]
DIV12 = [[-3, 1, 1, -1, 1, -1, -1], [1, -3, 1, -1, -1, 1, -1], [1, 1, -3, 1, -1, -1, -1]]
KINDS = ["pairs", "turns", "extreme", "wide", "tiny", "huge"]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


def _field(kind, dims, rng):
    nx, ny, nz = dims
    i, j, k = (x.ravel() for x in np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"))
    i, j, k = (x.reshape(nx, ny, nz).transpose(2, 1, 0).ravel() for x in (i, j, k))
    x = rng.uniform(0.5, 1.5, i.size) * rng.choice([-1.0, 1.0], i.size)
    if kind == "pairs":
        x = np.where(i % 2 == 1, 2.0 ** 30, x)
    elif kind == "turns":
        x = np.where(i % 4 == 1, 2.0 ** 30, np.where(i % 4 == 3, -2.0 ** 30, x))
    elif kind == "extreme":
        x = (2 - 2.0 ** -52) * np.where((i + j + k) % 2 == 1, 1.0, -1.0)
    elif kind == "wide":
        x *= 10.0 ** rng.uniform(-30, 0, i.size)
    elif kind == "tiny":
        x *= 1e-300
    elif kind == "huge":
        x *= 1e303
    return x


def _at(x, dims, o):
    nx, ny, nz = dims
    v = x.reshape(nz, ny, nx).astype(np.longdouble)
    return v[1 + o[2]:nz - 1 + o[2], 1 + o[1]:ny - 1 + o[1], 1 + o[0]:nx - 1 + o[0]]


def _nb6(x, dims):
    """Sum of the six axis neighbours, and of the magnitudes of its three pairs."""
    s = [_at(x, dims, o) + _at(x, dims, [-c for c in o]) for o in KUHN[:3]]
    return sum(s), sum(abs(v) for v in s)


def _div(x, dims, d):
    """12 Div_d, and the sum of |weight| |pair|."""
    t = [(w, _at(x, dims, o) - _at(x, dims, [-c for c in o])) for w, o in zip(DIV12[d], KUHN)]
    return sum(w * v for w, v in t), sum(abs(w) * abs(v) for w, v in t)


def _mesh(pkg, name, level):
    macro = macro_by_name(name)
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=1)
    nx, ny, nz = mesh.dims()
    k, j, i = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    regular = ((mesh.node_flags() & 7) == 3).reshape(nz, ny, nx)
    first = regular & ((i + j + k) % 4 == 0)  # a sweep's first colour reads the state as given
    inner = (slice(1, -1),) * 3
    h = np.longdouble(1.0) / (1 << level)
    return mesh, (nx, ny, nz), regular[inner], first[inner], h, h * h / 12, (h ** 3 / 6) ** (np.longdouble(2) / 3) * h / 12


def _check(got, want, size, where, dims):
    nx, ny, nz = dims
    g = got.reshape(nz, ny, nx)[1:-1, 1:-1, 1:-1]
    assert where.any()
    err = np.abs(g - want) - (16 * U * size + 64 * np.longdouble(2.0) ** -1074)
    assert np.all(err[where] <= 0), ((err[where] > 0).sum(), float(np.max(np.abs(g - want)[where] / np.maximum(size[where], 1e-320)) / U))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("name,level", [("cube", 4), ("channel", 2), ("partial", 3)])
def test_divergence_rows(pkg, name, level, kind):
    mesh, dims, regular, first, h, b, c = _mesh(pkg, name, level)
    n, rng = mesh.num_nodes(), np.random.default_rng(6)
    zero, fl = np.zeros(n), mesh.node_flags()
    x = np.where(fl & 1, _field(kind, dims, rng), 0.0)
    # the residual's gradient rows: K (0, p)
    ku, _ = mesh.apply_operator(np.zeros((n, 3)), x)
    # the velocity right-hand side f - B^T p
    mesh.level_field(level, "F", 0, np.zeros((n, 3)))
    mesh.level_field(level, "P", 0, x)
    mesh.level_op(level, "vel_rhs")
    ru = mesh.level_field(level, "RU")
    for d in range(3):
        val, size = _div(x, dims, d)
        _check(ku[:, d], -b * val, b * size, regular, dims)
        _check(ru[:, d], b * val, b * size, regular, dims)
    # one pressure colour from p = 0: p = w (B u - g), u_d = x in one component at a time
    w = np.longdouble(mesh.options.omega) / (6 * c)
    x = np.where(fl & 2, x, 0.0)
    for d in range(3):
        u = np.zeros((n, 3))
        u[:, d] = x
        mesh.level_field(level, "U", 0, u)
        mesh.level_field(level, "P", 0, zero)
        mesh.level_field(level, "G", 0, zero)
        mesh.level_op(level, "pres_sweep_f")
        val, size = _div(x, dims, d)
        _check(mesh.level_field(level, "P"), w * b * val, w * b * size, first, dims)
    mesh.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("name,level", [("cube", 4), ("channel", 2), ("partial", 3)])
def test_laplacian_rows(pkg, name, level, kind):
    mesh, dims, regular, first, h, b, c = _mesh(pkg, name, level)
    n, rng = mesh.num_nodes(), np.random.default_rng(7)
    x = np.where(mesh.node_flags() & 2, _field(kind, dims, rng), 0.0)
    nb, size = _nb6(x, dims)
    xc = _at(x, dims, (0, 0, 0))
    # the residual's Laplacian rows: K (u, 0)
    u = np.zeros((n, 3))
    u[:, 1] = x
    ku, _ = mesh.apply_operator(u, np.zeros(n))
    _check(ku[:, 1], h * (6 * xc - nb), h * (6 * abs(xc) + size), regular, dims)
    # one velocity colour from RU = 0: u = sum of the neighbours / 6
    mesh.level_field(level, "U", 0, u)
    mesh.level_field(level, "RU", 0, np.zeros((n, 3)))
    mesh.level_op(level, "vel_forward")
    _check(mesh.level_field(level, "U")[:, 1], nb / 6, size / 6, first, dims)
    # one pressure colour from u = 0, g = 0: p - w C p
    mesh.level_field(level, "U", 0, np.zeros((n, 3)))
    mesh.level_field(level, "P", 0, x)
    mesh.level_field(level, "G", 0, np.zeros(n))
    mesh.level_op(level, "pres_sweep_f")
    w = np.longdouble(mesh.options.omega) / 6
    _check(mesh.level_field(level, "P"), xc - w * (6 * xc - nb), abs(xc) + w * (6 * abs(xc) + size), first, dims)
    mesh.close()
