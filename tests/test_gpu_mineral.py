"""The mineral a dissolution pass takes, with one rate and with a rate field,
across periodic sides and across the cuts of a split lattice.

The pass after initialisation is held to w_j k u / W_s summed over the fluid
neighbours in extended precision: eight products and their sum to 2^-47 each,
10 x 2^-47 = 7e-14 of the amount, and the FP64 rounding of the difference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W36 = [16, 4, 4, 4, 4, 1, 1, 1, 1]
NX, NY, K = 131, 97, 0.3
LD = np.longdouble


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_02708_gb300 as pkg
    return pkg


def _case(field, mineral):
    rng = np.random.default_rng(7)
    solid = rng.random((NY, NX)) < 0.5
    u = (rng.uniform(0.1, 1.0, (NY, NX)) * ~solid).astype(np.float32).astype(np.float64)
    kf = rng.uniform(0.1, 0.5, (NY, NX)).astype(np.float32).astype(np.float64)
    return dict(solid=solid, vel=np.zeros((2, NY, NX)), u0=u, react_mode=1, k=K, dissolution=True,
                k_field=kf if field else None, mineral=np.full((NY, NX), mineral))


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("field", [False, True])
def test_first_pass(gb, precision, field):
    kw = _case(field, 2.0)
    solid, u, k = kw["solid"], kw["u0"].astype(LD), kw["k_field"] if field else K
    lat = gb.LBM(NX, NY, 0.8, precision=precision, **kw)
    ws = sum(W36[i] * np.roll(solid, (cy, cx), (0, 1)) for i, (cx, cy) in enumerate(C) if i)
    r = k * u / np.maximum(ws, 1)
    take = sum(W36[i] * np.roll(r, (cy, cx), (0, 1)) for i, (cx, cy) in enumerate(C) if i)
    got = (LD(2) - lat.mineral())[solid]
    assert np.abs(got - take[solid]).max() <= 7e-14 * float(take.max()) + 2.0 ** -53


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("edges", [(1, 2, 0, 0), (0, 0, 1, 1)])
def test_rate_field_across_cuts(gb, precision, edges):
    from paper_1601_02708_gb300.partition import SlabLattice
    kw = _case(True, 0.4)
    whole = gb.LBM(NX, NY, 0.8, edges=edges, precision=precision, **kw)
    split = SlabLattice(NX, NY, 0.8, parts=3, edges=edges, precision=precision, **kw)
    ud = np.ones(2 * (NX + NY))
    new = kw["k_field"][::-1].copy()
    for _ in range(2):
        for lat in (whole, split):
            lat.substeps(9, 1, ud, ud)
        assert np.array_equal(split.populations(), whole.populations())
        assert np.array_equal(split.mineral(), whole.mineral())
        whole.set_rate_field(new)
        for s in split.slabs:
            s.set_rate_field(new[s.y0:s.y1])
    assert whole.diagnostics()["flips"] > 50
