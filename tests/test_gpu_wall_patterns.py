"""The maximum-entropy wall solve over every kind of neighbourhood: a mask of
independent random nodes holds walls, corners, tips and one-node pores in all
orientations, and one step from a random state is compared with the same step
in extended precision, at magnitudes inside and outside the range of the
polynomial solve.  (The FP64 oracle solves for the logarithm of the root, so
at 1e-26 its own populations are 3e-14 off; the CPU test bounds that.)

Tolerances relative to max|f|: one step rounds a population to FP32 about ten
times (pull, moments, collision), so 10 x 2^-24 = 6e-7, taken twice for the
sum's condition; FP64 likewise 20 x 2^-53 = 2.2e-15, times 12 because an
unknown carries up to twelve powers of the root."""
import numpy as np
import pytest

C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W36 = [16, 4, 4, 4, 4, 1, 1, 1, 1]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
NX, NY, TAU = 131, 97, 0.9
LD = np.longdouble


def _inputs(scale):
    rng = np.random.default_rng(5)
    solid = (rng.random((NY, NX)) < 0.4).astype(np.uint8)
    patterns = sum(np.roll(solid, s, (0, 1)).astype(int) << k for k, s in enumerate(
        [(0, 1), (1, 0), (0, -1), (-1, 0), (1, 1), (1, -1), (-1, -1), (-1, 1)]))
    assert len(np.unique(patterns[solid == 0])) == 256
    vel = 0.05 * rng.uniform(-1, 1, (2, NY, NX)) * (solid == 0)
    u0 = scale * rng.uniform(0.2, 1.0, (NY, NX)) * (solid == 0)
    return dict(edges=(0, 0, 0, 0), solid=solid, vel=vel, u0=u0)


def _extended(kw):
    """Populations after one step in extended precision, [9, NY, NX]."""
    w = [LD(k) / 36 for k in W36]
    vx, vy = kw["vel"].astype(LD)
    u = kw["u0"].astype(LD)
    solid = kw["solid"] != 0

    def collide(f, u):
        out = []
        for i, (cx, cy) in enumerate(C):
            ev = cx * vx + cy * vy
            eq = w[i] * u * (1 + 3 * ev + LD(4.5) * ev * ev - LD(1.5) * (vx * vx + vy * vy))
            out.append(eq if f is None else f[i] + (eq - f[i]) / LD(TAU))
        return np.stack(out)

    f = collide(collide(None, u), u)  # the equilibrium, collided once
    up = [np.roll(solid, (cy, cx), (0, 1)) for cx, cy in C]
    g = np.stack([np.where(up[i], f[OPP[i]], np.roll(f[i], (cy, cx), (0, 1)))
                  for i, (cx, cy) in enumerate(C)])
    for y, x in zip(*np.nonzero(~solid & np.any(up[1:], 0))):
        link = [i for i in range(1, 9) if up[i][y, x]]
        m = -np.sum([W36[i] * np.array(C[i]) for i in link], 0)
        d = [-int(np.dot(c, m)) for c in C]
        neg = [i for i in link if d[i] > 0]
        if not neg:
            continue
        T = -sum(d[i] * g[i, y, x] for i in range(9) if i not in neg)
        if T > 0:
            # sum 36 w d t^d = 36 e T: bracketed, then Newton
            e = np.exp(LD(1))
            lo = hi = LD(1)
            p = lambda t: sum(w[i] * d[i] * t ** d[i] for i in neg) - e * T
            while p(lo) > 0:
                lo /= 4
            while p(hi) < 0:
                hi *= 4
            t = hi  # p is convex and increasing: Newton descends monotonically
            for _ in range(200):
                step = p(t) / sum(w[i] * d[i] ** 2 * t ** (d[i] - 1) for i in neg)
                t -= step
                if abs(step) <= LD(1e-18) * t:
                    break
        for i in neg:
            g[i, y, x] = w[i] / e * t ** d[i] if T > 0 else 0
    return collide(g, g.sum(0))


@pytest.mark.parametrize("scale,off", [(1.0, 3e-15), (1e-26, 1e-13)])
def test_extended_step_agrees_with_the_oracle(oracle_mod, scale, off):
    """The reference of the GPU test against the oracle (its logarithm of a
    root near 1e-26 is about 60, so its rounding is 60 times larger)."""
    kw = _inputs(scale)
    ref = oracle_mod.LBMOracle(NX, NY, TAU, walls="maxent", **kw)
    ref.substeps(1, 1)
    fluid = kw["solid"] == 0
    a, b = _extended(kw)[:, fluid], ref.fpost()[:, fluid]
    assert np.abs(a - b).max() <= off * np.abs(a).max()


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1.0, 1e-20, 1e-26, 1e26])
@pytest.mark.parametrize("prec,tol", [(32, 1.2e-6), (64, 2.7e-14)])
def test_every_neighbourhood(prec, tol, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBM
    kw = _inputs(scale)
    lat = LBM(NX, NY, TAU, precision=prec, walls="maxent", **kw)
    lat.substeps(1, 1)
    f, fr = lat.populations(), _extended(kw).astype(np.float64)
    fluid = kw["solid"] == 0
    assert np.abs(f - fr)[:, fluid].max() <= tol * np.abs(fr[:, fluid]).max()
    assert lat.diagnostics()["newton_fail"] == 0
