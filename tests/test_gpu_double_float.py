"""What the double-float forms of the FP32 lattice carry: the pore wall's root
and the boundary solves, element by element against extended precision.  A
relaxation time of 1e30 leaves the moving populations unchanged by the
collision, so a step's stored populations are the streamed ones and the solves'
results, rounded to FP32 once.

Tolerances.  A population is the FP32 number nearest to a value within 1.2e-9
(wall: the remainder of the last Newton step, twelve powers of it) or 2^-48 of
the largest term of its sum (sides: at least a thousandth of that term) of the
exact one: 2^-24 + 1.2e-9 = 6.1e-8 relative."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W36 = [16, 4, 4, 4, 4, 1, 1, 1, 1]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
LD = np.longdouble
ULP = 6.1e-8


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_02708_gb300 as pkg
    return pkg


def with_populations(lat, f):
    """The lattice with the FP32 populations f [9, ny, nx] in place of its own,
    and their images beyond the sides as on a periodic lattice."""
    _, ny, nx = f.shape
    rows, pitch = max(ny + 2, 10), max((nx + 47) // 32 * 32, 160)
    blob = lat.save(np.zeros(lat.state_bytes(), np.uint8))
    planes = blob[256:256 + 9 * rows * pitch * 4].view(np.float32).reshape(9, rows, pitch)
    planes[:, :ny + 2, 7:nx + 9] = np.pad(f, ((0, 0), (1, 1), (1, 1)), mode="wrap")
    lat.restore(blob)
    assert np.array_equal(lat.populations(), f)
    return lat


def streamed(f, solid):
    """Populations after streaming and bounce-back on a periodic lattice, and
    whether each came from a solid node."""
    up = np.stack([np.roll(solid, (cy, cx), (0, 1)) for cx, cy in C])
    g = np.stack([np.where(up[i], f[OPP[i]], np.roll(f[i], (cy, cx), (0, 1)))
                  for i, (cx, cy) in enumerate(C)])
    return g, up


def wall_solve(g, link):
    """The unknowns of a wall node in extended precision: {i: value} and T."""
    m = -np.sum([W36[i] * np.array(C[i]) for i in link], 0)
    d = [-int(np.dot(c, m)) for c in C]
    neg = [i for i in link if d[i] > 0]
    if not neg:
        return {}, LD(0)
    T = -sum(LD(d[i]) * LD(g[i]) for i in range(9) if i not in neg)
    if not T > 0:
        return {i: LD(0) for i in neg}, T
    e = np.exp(LD(1))
    w = [LD(k) / 36 for k in W36]
    x = LD(0)  # log t: Newton on the convex log p converges from any start
    goal = np.log(e * T)
    for _ in range(200):
        terms = {i: w[i] * d[i] * np.exp(d[i] * x) for i in neg}
        p = sum(terms.values())
        step = (np.log(p) - goal) * p / sum(d[i] * v for i, v in terms.items())
        x -= step
        if abs(step) < LD(1e-17):
            break
    t = np.exp(x)
    return {i: w[i] / e * t ** d[i] for i in neg}, T


@pytest.mark.parametrize("kernel", ["tma", "generic"])
def test_wall_root(gb, kernel):
    nx, ny = 131, 97
    rng = np.random.default_rng(5)
    solid = rng.random((ny, nx)) < 0.4
    f = rng.uniform(0.01, 1.0, (9, ny, nx)).astype(np.float32) * ~solid
    lat = gb.LBM(nx, ny, 1e30, solid=solid, vel=np.zeros((2, ny, nx)), u0=np.zeros((ny, nx)), walls="maxent")
    lat.set_kernel(kernel)
    with_populations(lat, f).substeps(1, 1)
    got, (g, up) = lat.populations(), streamed(f, solid)
    worst, noroot = 0.0, 0
    for y, x in zip(*np.nonzero(~solid)):
        link = [i for i in range(1, 9) if up[i, y, x]]
        want, T = wall_solve(g[:, y, x], link) if link else ({}, 0)
        noroot += T < 0
        for i in range(1, 9):
            if i in want:
                worst = max(worst, abs(got[i, y, x] - want[i]) / want[i] if want[i] > 0 else got[i, y, x])
            else:
                assert got[i, y, x] == g[i, y, x]
    assert worst <= ULP
    assert lat.diagnostics()["bc_infeasible"] == noroot > 0


@pytest.mark.parametrize("kernel", ["tma", "generic"])
def test_side_solves(gb, kernel):
    nx, ny = 70, 45
    rng = np.random.default_rng(6)
    f = rng.uniform(0.01, 1.0, (9, ny, nx)).astype(np.float32)
    lat = gb.LBM(nx, ny, 1e30, edges=(1, 2, 0, 0), vel=np.zeros((2, ny, nx)), u0=np.zeros((ny, nx)))
    lat.set_kernel(kernel)
    ud, q = rng.uniform(6.0, 9.0, 2 * (nx + ny)), rng.uniform(-1.0, 0.01, 2 * (nx + ny))
    with_populations(lat, f).substeps(1, 1, ud, ud, q)
    got, g = lat.populations(), streamed(f, np.zeros((ny, nx), bool))[0].astype(LD)
    for x, unknown, first in ((0, (1, 5, 8), 0), (nx - 1, (3, 6, 7), ny)):
        for y in range(ny):
            known = [i for i in range(9) if i not in unknown]
            if x == 0:
                rest = LD(ud[first + y]) - sum(g[i, y, x] for i in known)
            else:
                rest = sum(C[i][0] * g[i, y, x] for i in known) - LD(q[first + y])
            assert rest > 0
            for i in unknown:
                want = rest * W36[i] / 6
                assert abs(got[i, y, x] - want) <= ULP * want
            for i in known[1:]:
                assert got[i, y, x] == g[i, y, x]


# One solid node beside a fluid one: the side it lies on, and the populations of
# the flux sum in the order of their directions.  Terms near one and near 2^-25
# cancel, and what is left is below 2^-48 of the largest.
CANCEL = [
    ("E", ["0x1.00001p-24", "0x1p+0", "0x1p+0", "0x1.00001p-24", "0x1p-49"]),
    ("W", ["0x1p+0", "0x1p-50", "0x1.7ffff6p-4", "0x1.4p-25", "0x1.18p+0"]),
    ("N", ["0x1.4p-49", "0x1.0008p+0", "0x1.fff00cp-1", "0x1.000004p+0", "0x1.000002p+0"]),
    ("S", ["0x1p-51", "0x1p-26", "0x1.00004p+0", "0x1p+0", "0x1.01p-18"]),
]


@pytest.mark.parametrize("kernel", ["tma", "generic"])
def test_wall_flux_that_cancels(gb, kernel):
    """The root, and whether there is one, where the flux sum cancels."""
    nx, ny = 64, 40
    to = {"E": (1, 0), "W": (-1, 0), "N": (0, 1), "S": (0, -1)}
    solid = np.zeros((ny, nx), bool)
    f = np.full((9, ny, nx), 0.5, np.float32)
    nodes = []
    for k, (side, values) in enumerate(CANCEL):
        x, y, (sx, sy) = 8 + 12 * k, 20, to[side]
        solid[y + sy, x + sx] = True
        nodes.append((x, y))
        terms = [i for i in range(1, 9) if C[i][0] * sx + C[i][1] * sy and C[i] != (-sx, -sy)]
        for i, v in zip(terms, values):
            f[i, y - C[i][1], x - C[i][0]] = float.fromhex(v)
    f *= ~solid
    lat = gb.LBM(nx, ny, 1e30, solid=solid, vel=np.zeros((2, ny, nx)), u0=np.zeros((ny, nx)), walls="maxent")
    lat.set_kernel(kernel)
    with_populations(lat, f).substeps(1, 1)
    got, (g, up) = lat.populations(), streamed(f, solid)
    noroot = 0
    for y, x in zip(*np.nonzero(~solid)):
        link = [i for i in range(1, 9) if up[i, y, x]]
        want, T = wall_solve(g[:, y, x], link) if link else ({}, 0)
        noroot += T < 0
        if (x, y) in nodes:
            assert 0 < abs(T) < 1e-14
        for i, v in want.items():
            if T > 0:
                assert abs(got[i, y, x] - v) <= ULP * v
            else:  # zero, and what the collision adds: w u / tau
                assert 0 <= got[i, y, x] <= 1e-30
    assert lat.diagnostics()["bc_infeasible"] == noroot == 1
