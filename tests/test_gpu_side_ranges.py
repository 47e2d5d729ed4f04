"""Side solves of the FP32 lattice where double-float does not hold the data:
tiny and huge values, and differences far smaller than their terms.  Against
extended precision, element by element; the populations lie within 2^7 of each
other, so FP64 holds their sums exactly, its difference from the edge data too
(they are nearly equal, or it is rounded to 2^-53 of itself), and the unknowns
are rounded to FP32 once: 6.1e-8 relative."""
import numpy as np
import pytest

from test_gpu_double_float import C, LD, ULP, W36, gb, streamed, with_populations  # noqa: F401

pytestmark = pytest.mark.gpu

NX, NY = 70, 45


@pytest.mark.parametrize("kernel", ["tma", "generic"])
@pytest.mark.parametrize("exponent,cancel", [(-82, False), (-110, False), (100, False), (0, True), (-85, True)])
def test_side_solves(gb, exponent, cancel, kernel):  # noqa: F811
    rng = np.random.default_rng(exponent + 200)
    f = np.ldexp(rng.uniform(0.01, 1.0, (9, NY, NX)), exponent).astype(np.float32)
    ud = np.ldexp(rng.uniform(6.0, 9.0, 2 * (NX + NY)), exponent)
    q = np.ldexp(rng.uniform(-1.0, 0.01, 2 * (NX + NY)), exponent)
    g = streamed(f, np.zeros((NY, NX), bool))[0].astype(LD)
    unknown = {0: (1, 5, 8), NX - 1: (3, 6, 7)}
    known = {x: [i for i in range(9) if i not in unknown[x]] for x in unknown}
    if cancel:
        for y in range(NY):
            part = np.ldexp(1.0, -11 - y % 20) * (-1) ** (y // 20)
            ud[y] = float(sum(g[i, y, 0] for i in known[0])) * (1 + part)
            q[NY + y] = float(sum(C[i][0] * g[i, y, NX - 1] for i in known[NX - 1])) * (1 - part)
    lat = gb.LBM(NX, NY, 1e30, edges=(1, 2, 0, 0), vel=np.zeros((2, NY, NX)), u0=np.zeros((NY, NX)))
    lat.set_kernel(kernel)
    with_populations(lat, f).substeps(1, 1, ud, ud, q)
    got, low = lat.populations(), 0
    for x in unknown:
        for y in range(NY):
            if x == 0:
                rest = LD(ud[y]) - sum(g[i, y, x] for i in known[x])
            else:
                rest = sum(C[i][0] * g[i, y, x] for i in known[x]) - LD(q[NY + y])
            low += rest < 0
            for i in unknown[x]:
                want = rest * W36[i] / 6 if x == 0 or rest > 0 else LD(0)
                # (what the collision adds is below 1e-29 of the largest population)
                assert abs(got[i, y, x] - want) <= ULP * abs(want) + np.ldexp(1e-29, exponent)
            for i in known[x][1:]:
                assert got[i, y, x] == g[i, y, x]
    assert lat.diagnostics()["bc_infeasible"] == low
    assert (low > 0) == cancel
