"""Mass of a closed FP64 lattice over thousands of steps: every collision leaves
(1 - k) u in the stored populations, so with periodic sides and bounce-back walls
the total follows (1 - k)^n.

Bound: the sum of a node's populations is off by the roundings of one step, at
most about 2^-53 of u and as often up as down.  Where a steady state repeats them
in every step, n of them add up at a node, and over N nodes of either sign the
total is off by n 2^-53 / sqrt(N), 6e-15 here; the bound is three times that.
(Weights that sum to 1 - 5.6e-17, as 4/9, 1/9 and 1/36 do in FP64, cost
n omega 5.6e-17, 2.2e-13 and more.)"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY, STEPS = 96, 64, 4000


def _mass(lat, solid):
    return math.fsum(lat.populations()[:, solid == 0].ravel())


@pytest.mark.parametrize("shape", ["alone", "batch"])
@pytest.mark.parametrize("tau,k", [(0.6, 0.0), (0.7, 0.0), (1.0, 0.0), (3.0, 0.0), (0.8, 2.0**-12)])
def test_mass_of_a_closed_lattice(tau, k, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBM, LBMBatch
    rng, stream = np.random.default_rng(3), torch.cuda.Stream()
    solid = (rng.random((NY, NX)) < 0.1).astype(np.uint8)
    vel = np.where(solid, 0.0, 0.02 * rng.standard_normal((2, NY, NX)))
    lat = LBM(NX, NY, tau, precision=64, solid=solid, vel=vel, u0=np.where(solid, 0.0, rng.random((NY, NX))),
              react_mode=2 if k else 0, k=k, stream=stream.cuda_stream)
    before = _mass(lat, solid)
    run = lat if shape == "alone" else LBMBatch([lat])
    for _ in range(STEPS // 500):
        run.substeps(500)
    want = before * (1.0 - k) ** STEPS
    assert abs(_mass(lat, solid) - want) <= 2e-14 * want
