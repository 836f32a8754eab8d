"""FP64 stencils in aligned integers: K (u, p) of the residual kernel at
regular nodes against the closed-form stencils in extended precision, over
fields of one and of many magnitudes, near the ends of the FP64 range (where
the kernel takes FP64 operations), of zeros, and with infinities and NaN.

Tolerance: 16 u (|K| |x|) per row with u = 2^-53.  A stencil sum carries at
most 18 cut-off units of 2^-5 u and one rounding, below 1.1 u of its largest
value; the row then rounds at most five products and three sums, and the
level's scale factors carry a few u of their own."""
import numpy as np
import pytest

from tests.helpers import macro_by_name

pytestmark = pytest.mark.gpu

KINDS = ["normal", "wide", "mixed", "tiny", "huge", "sparse"]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_1511_02134_gb300 as p
    return p


def _field(kind, shape, rng):
    x = rng.standard_normal(shape)
    if kind == "wide":
        x *= 10.0 ** rng.uniform(-30, 0, shape)
    elif kind == "mixed":
        x = np.where(rng.random(shape) < 0.3, 0.0, x) * np.where(rng.random(shape) < 0.5, 1.0, 1e-9)
    elif kind == "tiny":
        x *= 1e-300
    elif kind == "huge":
        x *= 1e303
    elif kind == "sparse":
        x = np.where(rng.random(shape) < 0.01, x, 0.0)
    return x


KUHN = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, 1, 1)]
DIV12 = [[-3, 1, 1, -1, 1, -1, -1], [1, -3, 1, -1, -1, 1, -1], [1, 1, -3, 1, -1, -1, -1]]


def _closed_form(u, p, dims, h):
    """K (u, p) and |K| |(u, p)| on interior positions, extended precision (nu = 1, delta = 1/12)."""
    nx, ny, nz = dims
    ext = np.longdouble
    U = [u[:, d].reshape(nz, ny, nx).astype(ext) for d in range(3)]
    P = p.reshape(nz, ny, nx).astype(ext)

    def at(x, o, s):
        i, j, k = (s * c for c in o)
        return x[1 + k:nz - 1 + k, 1 + j:ny - 1 + j, 1 + i:nx - 1 + i]

    def lap(x):
        nb = [at(x, o, s) for o in KUHN[:3] for s in (1, -1)]
        c = at(x, (0, 0, 0), 1)
        return 6 * c - sum(nb), 6 * abs(c) + sum(abs(v) for v in nb)

    def div(x, d):
        t = [(w, at(x, o, 1), at(x, o, -1)) for w, o in zip(DIV12[d], KUHN)]
        return sum(w * (a - b) for w, a, b in t), sum(abs(w) * (abs(a) + abs(b)) for w, a, b in t)

    h = ext(h)
    b, c = h * h / 12, (h ** 3 / 6) ** (ext(2) / 3) * h / 12
    val, mag = [], []
    for d in range(3):
        (a, am), (g, gm) = lap(U[d]), div(P, d)
        val.append(h * a - b * g)
        mag.append(h * am + b * gm)
    dv = [div(U[d], d) for d in range(3)]
    (q, qm) = lap(P)
    val.append(b * sum(v for v, _ in dv) - c * q)
    mag.append(b * sum(m for _, m in dv) + c * qm)
    return val, mag


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("name,level", [("cube", 4), ("channel", 2), ("partial", 3)])
def test_regular_rows_against_extended_precision(pkg, name, level, kind):
    macro = macro_by_name(name)
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, level, coarsest_level=1)
    n, dims, fl = mesh.num_nodes(), mesh.dims(), mesh.node_flags()
    rng = np.random.default_rng(4)
    u, p = _field(kind, (n, 3), rng), _field(kind, n, rng)
    u[(fl & 2) == 0] = 0.0
    p[(fl & 1) == 0] = 0.0
    ku, kp = mesh.apply_operator(u, p)
    val, mag = _closed_form(u, p, dims, 1.0 / (1 << level))
    nx, ny, nz = dims
    inner = lambda x: x.reshape(nz, ny, nx)[1:-1, 1:-1, 1:-1]  # noqa: E731
    regular = inner((fl & 7) == 3)
    assert regular.any()
    for d, got in enumerate([ku[:, 0], ku[:, 1], ku[:, 2], kp]):
        # (subnormal results round at 2^-1074)
        err = np.abs(inner(got) - val[d]) - (16 * 2.0 ** -53 * mag[d] + 64 * 2.0 ** -1074)
        assert np.all(err[regular] <= 0), (d, (err[regular] > 0).sum())
    mesh.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_not_finite_values_reach_every_row_that_reads_them(pkg, value):
    macro = macro_by_name("cube")
    mesh = pkg.Mesh(macro.vertices, macro.tets, macro.bc_flags, 3, coarsest_level=2)
    n, nx = mesh.num_nodes(), mesh.dims()[0]
    u, p = np.zeros((n, 3)), np.zeros(n)
    c = 4 + nx * (4 + nx * 4)
    u[c, 1] = value
    ku, kp = mesh.apply_operator(u, p)
    bad = ~np.isfinite(ku[:, 1])
    near = {c + s * o for s in (0, 1, -1) for o in (1, nx, nx * nx)}
    assert set(np.where(bad)[0]) == near
    diag = {c + s * o for s in (1, -1) for o in (1, nx, nx * nx, 1 + nx, nx + nx * nx, 1 + nx * nx, 1 + nx + nx * nx)}
    assert set(np.where(~np.isfinite(kp))[0]) == diag
    mesh.close()
