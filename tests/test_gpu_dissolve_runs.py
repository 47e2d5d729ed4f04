"""Dissolution passes in which many adjacent nodes flip at once, so that nodes
are examined while their neighbours turn fluid and while nodes behind them are
put on the surface list: masks, flip counts and minerals against the oracle at
every few steps, on one lattice and as a batch member.  FP64: masks are equal
and minerals within a rounding of each of the at most 8 terms of 60 passes,
8 x 60 x 2^-53 = 5e-14."""
import numpy as np
import pytest

from paper_1601_02708_gb300 import inputs

pytestmark = pytest.mark.gpu


def _case(nx, ny, edges):
    rng = np.random.default_rng(nx)
    solid = (rng.random((ny, nx)) < 0.55).astype(np.uint8)
    solid[ny // 4:3 * ny // 4, nx // 4:3 * nx // 4] = 1  # a block that dissolves from outside
    solid[:, [0, -1]] = 0
    # equal minerals flip together, the random half one after another
    mineral = np.where(rng.random((ny, nx)) < 0.5, 0.02, rng.uniform(0.001, 0.03, (ny, nx)))
    u0 = np.where(solid != 0, 0.0, rng.uniform(0.5, 1.0, (ny, nx)))
    return dict(edges=edges, solid=solid, vel=np.zeros((2, ny, nx)), u0=u0, react_mode=1, k=0.05,
                dissolution=True, mineral=mineral)


@pytest.mark.parametrize("shape,edges", [((97, 61), (1, 2, 0, 0)), ((33, 40), (0, 0, 0, 0)),
                                         ((200, 34), (1, 1, 1, 1))])
@pytest.mark.parametrize("batch", [False, True])
def test_many_flips_in_one_pass(oracle_mod, shape, edges, batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBM, LBMBatch
    nx, ny = shape
    kw = _case(nx, ny, edges)
    ud = inputs.edge_array(nx, ny, 1.0, 1.0, 1.0, 1.0)
    now, ahead = (oracle_mod.LBMOracle(nx, ny, 0.8, **kw) for _ in range(2))
    s = torch.cuda.Stream()
    lat = LBM(nx, ny, 0.8, precision=64, stream=s.cuda_stream, **kw)
    run = LBMBatch([lat]) if batch else None
    ahead.substeps(1, 1, ud, ud)  # the library decides a flip one step ahead
    most = before = 0
    for n in (1, 4, 7, 18, 30):
        if batch:
            run.substeps(n, 1, [ud], [ud])
        else:
            lat.substeps(n, 1, ud, ud)
        now.substeps(n, 1, ud, ud)
        ahead.substeps(n, 1, ud, ud)
        assert np.array_equal(lat.solid(), now.solid())
        assert np.array_equal(lat.flip_steps(), now.flip_steps())
        flips = lat.diagnostics()["flips"]
        assert flips == ahead.diag()["flips"]
        left = ahead.solid() != 0
        assert np.abs(lat.mineral() - ahead.mineral())[left].max() <= 5e-14
        most, before = max(most, flips - before), flips
    assert most > 50


@pytest.mark.parametrize("shape", [(33, 40), (400, 300)])
@pytest.mark.parametrize("precision", [32, 64])
def test_restored_solids_have_no_shares(oracle_mod, shape, precision):
    """Nodes that were fluid, with shares, and are solid again after a restore
    flip anew beside neighbours examined in the same pass: every run from the
    restored state ends in the same bits, and the FP64 mask is the oracle's."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBM
    nx, ny = shape
    kw = _case(nx, ny, (1, 1, 1, 1))
    ud = inputs.edge_array(nx, ny, 1.0, 1.0, 1.0, 1.0)
    lat = LBM(nx, ny, 0.8, precision=precision, **kw)
    start = lat.save()
    n = 40
    runs = []
    for _ in range(6):
        lat.restore(start)
        lat.substeps(n, 1, ud, ud)
        runs.append((lat.solid(), lat.mineral(), lat.flip_steps()))
    assert lat.diagnostics()["flips"] > 200
    for run in runs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(run, runs[0]))
    if precision == 64:
        ref = oracle_mod.LBMOracle(nx, ny, 0.8, **kw)
        ref.substeps(n, 1, ud, ud)
        assert np.array_equal(runs[0][0], ref.solid())
