"""The continuum solve is linear: data scaled by a power of two, as far as
squares of the data stay in FP64's range, give the scaled solution in as many
iterations.  (The scaling is exact, so the sums differ in nothing but their
exponents.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-440, -330, -200, 200, 330, 440])
@pytest.mark.parametrize("nex,ney", [(37, 11), (151, 149)])
def test_scaled_data(nex, ney, exponent):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300.fem import FEM
    rng = np.random.default_rng(nex)
    nxn = nex + 1
    dirichlet = [j * nxn for j in range(ney + 1)]
    d0 = rng.uniform(0, 1, nxn * (ney + 1))
    vals = rng.uniform(0, 2, len(dirichlet))
    out = []
    for e in (0, exponent):
        g = FEM(nex=nex, ney=ney, x0=0.0, y0=0.0, hx=0.02, hy=0.03, D=1e-3, v=(0.4, -0.15), theta=0.5,
                dt=0.01, supg=True, dirichlet=dirichlet, d0=np.ldexp(d0, e))
        for _ in range(2):
            g.step(np.ldexp(vals, e))
        out.append((np.ldexp(g.get(), -e), g.solver_info()[0]))
    (want, n), (got, m) = out
    assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
    assert abs(m - n) <= 1


@pytest.mark.parametrize("nex,ney", [(37, 11), (700, 330)])
def test_solve_cut_short(nex, ney):
    """By tiles and over the nodes in global memory: a solve stopped by max_iter
    is an error that tells its iterations; with the default limit it converges."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBMError
    from paper_1601_02708_gb300.fem import FEM
    rng = np.random.default_rng(3)
    nxn = nex + 1
    kw = dict(nex=nex, ney=ney, x0=0.0, y0=0.0, hx=0.02, hy=0.03, D=1e-3, v=(0.4, -0.15), theta=0.5,
              dt=0.01, supg=True, dirichlet=[j * nxn for j in range(ney + 1)],
              d0=rng.uniform(0, 1, nxn * (ney + 1)))
    vals = rng.uniform(0, 2, ney + 1)
    cut, full = FEM(max_iter=1, **kw), FEM(**kw)
    with pytest.raises(LBMError):
        cut.step(vals)
    assert cut.solver_info()[0] == 1
    full.step(vals)
    it, res = full.solver_info()
    assert 1 < it < 1000 and res <= 1e-12


def test_squares_below_the_normal_range():
    """Data whose residuals' squares leave FP64's normal range before the
    tolerance is met: the sums keep them, and the solution is within the
    tolerance times the scaled operator's condition (below 100)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300.fem import FEM
    nex, ney = 97, 53
    rng = np.random.default_rng(11)
    nxn = nex + 1
    dirichlet = [j * nxn for j in range(ney + 1)]
    d0, vals = rng.uniform(0, 1, nxn * (ney + 1)), rng.uniform(0, 2, len(dirichlet))
    out = []
    for e in (0, -505):
        g = FEM(nex=nex, ney=ney, x0=0.0, y0=0.0, hx=0.02, hy=0.03, D=1e-3, v=(0.4, -0.15), theta=0.5,
                dt=0.01, supg=True, dirichlet=dirichlet, d0=np.ldexp(d0, e), tol=1e-6)
        g.step(np.ldexp(vals, e))
        out.append(np.ldexp(g.get(), -e))
    assert np.abs(out[1] - out[0]).max() <= 2e-4
