"""A state restored where it was saved while a dissolution pass is due leaves
the run as it was, bit for bit: a slab's first pass after initialisation, and
the pass between the two halves of a step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY = 131, 57


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_02708_gb300 as pkg
    return pkg


def _case(edges):
    rng = np.random.default_rng(8)
    solid = (rng.random((NY, NX)) < 0.4).astype(np.uint8)
    if edges[0]:
        solid[:, [0, -1]] = 0
    return dict(edges=edges, solid=solid, vel=np.zeros((2, NY, NX)),
                u0=np.where(solid != 0, 0.0, rng.uniform(0.5, 1.0, (NY, NX))), react_mode=1, k=0.05,
                dissolution=True, mineral=rng.uniform(0.001, 0.02, (NY, NX)))


def _state(lat):
    return lat.populations(), lat.solid(), lat.mineral(), lat.flip_steps()


@pytest.mark.parametrize("where", ["device", "host"])
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("edges", [(1, 2, 0, 0), (0, 0, 1, 1)])
def test_before_the_first_pass_of_a_slab(gb, edges, precision, where):
    from paper_1601_02708_gb300.partition import SlabLattice
    ud = np.ones(2 * (NX + NY))
    runs = []
    for restored in (False, True):
        lat = SlabLattice(NX, NY, 0.8, parts=3, precision=precision, **_case(edges))
        for s in lat.slabs if restored else ():
            s.restore(s.save(None if where == "device" else np.zeros(s.state_bytes(), np.uint8)))
        runs.append([])
        for n in (1, 12):
            lat.substeps(n, 1, ud, ud)
            runs[-1] += _state(lat)
        lat.close()
    assert all(np.array_equal(a, b) for a, b in zip(*runs))
    assert (runs[0][-1] >= 0).any()


@pytest.mark.parametrize("where", ["device", "host"])
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("edges", [(1, 2, 0, 0), (0, 0, 1, 1), (0, 0, 0, 0)])
def test_between_the_halves_of_a_step(gb, edges, precision, where):
    from paper_1601_02708_gb300.partition import Slab
    ud = np.ones(2 * (NX + NY))
    runs = []
    for restored in (False, True):
        lat = Slab(NX, NY, 0.8, 0, NY, precision=precision, **_case(edges))  # the whole lattice
        lat.stage_edges(ud, ud)
        for j in range(1, 13):
            lat.stream(1, 1, True)
            if restored:
                lat.restore(lat.save(None if where == "device" else np.zeros(lat.state_bytes(), np.uint8)))
            lat.dissolve()
        runs.append(_state(lat))
        lat.close()
    assert all(np.array_equal(a, b) for a, b in zip(*runs))
    assert (runs[0][-1] >= 0).any()


@pytest.mark.parametrize("precision", [32, 64])
def test_run_resumed_in_fresh_slabs(gb, precision):
    """A run's states restored into slabs that have not stepped: they go on as it does."""
    from paper_1601_02708_gb300.partition import SlabLattice
    ud = np.ones(2 * (NX + NY))
    kw = _case((1, 2, 0, 0))
    run, fresh = (SlabLattice(NX, NY, 0.8, parts=3, precision=precision, **kw) for _ in range(2))
    run.substeps(12, 1, ud, ud)
    for a, b in zip(run.slabs, fresh.slabs):
        b.restore(a.save())
    for lat in (run, fresh):
        lat.substeps(9, 1, ud, ud)
    assert all(np.array_equal(a, b) for a, b in zip(_state(run), _state(fresh)))
    assert run.diagnostics()["flips"] == fresh.diagnostics()["flips"] > 0
