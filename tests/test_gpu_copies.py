"""States saved to and restored from device memory at every alignment, and edge
data of a batch of more members than one launch's list holds, from device and
host arrays: the bytes of the copies through host memory."""
import numpy as np
import pytest

from paper_1601_02708_gb300 import inputs

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, precision, seed=0, **kw):
    from paper_1601_02708_gb300 import LBM
    rng = np.random.default_rng(seed)
    solid = (rng.random((ny, nx)) < 0.3).astype(np.uint8)
    solid[:, [0, -1]] = 0
    return LBM(nx, ny, 0.8, edges=(1, 2, 0, 0), solid=solid, vel=np.zeros((2, ny, nx)),
               u0=np.where(solid, 0.0, rng.random((ny, nx))), react_mode=1, k=0.05, dissolution=True,
               mineral=rng.uniform(0.001, 0.02, (ny, nx)), precision=precision, **kw)


@pytest.mark.parametrize("offset", [0, 1, 4, 8, 16])
@pytest.mark.parametrize("shape,precision", [((33, 21), 32), ((130, 97), 64)])
def test_state_in_device_memory(shape, precision, offset):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lat = _lattice(*shape, precision)
    ud = inputs.edge_array(*shape, 1.0, 1.0, 1.0, 1.0)
    lat.substeps(12, 1, ud, ud)
    nb = lat.state_bytes()
    host = lat.save(np.zeros(nb, np.uint8))
    room = torch.full((nb + 64,), 7, dtype=torch.uint8, device="cuda")
    lat.save(room[offset:offset + nb])
    lat.synchronize()
    got = room.cpu().numpy()
    assert (got[:offset] == 7).all() and (got[offset + nb:] == 7).all()
    # the padding between sections is not written
    got = got[offset:offset + nb]
    assert np.array_equal(got[got != 7], host[got != 7])
    want = []
    for blob in (host, room[offset:offset + nb]):
        lat.restore(blob)
        lat.substeps(9, 1, ud, ud)
        want.append((lat.populations(), lat.solid(), lat.mineral(), lat.diagnostics()["steps"]))
    assert all(np.array_equal(a, b) for a, b in zip(*want))


@pytest.mark.parametrize("count", [3, 40])
def test_batch_edge_data(count):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02708_gb300 import LBMBatch
    out = []
    for where in ("host", "device", "mixed"):
        s = torch.cuda.Stream()
        m = [_lattice(33 + i % 5, 20 + i % 7, 32, i, stream=s.cuda_stream) for i in range(count)]
        edge = [np.random.default_rng(i).random(c.n_edge) for i, c in enumerate(m)]
        if where != "host":
            edge = [torch.from_numpy(e).cuda() if where == "device" or i % 2 else e
                    for i, e in enumerate(edge)]
        torch.cuda.synchronize()
        LBMBatch(m).substeps(4, 2, edge, edge)
        out.append([c.populations() for c in m])
    for other in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], other))


@pytest.mark.parametrize("offset", [0, 4, 16])
@pytest.mark.parametrize("shape,precision", [((33, 21), 32), ((130, 97), 64), ((517, 301), 32)])
def test_every_byte_of_a_state_is_written(shape, precision, offset):
    """Saved into buffers of two fills: a byte that keeps its fill in both was not
    written, and those are the ones that the copies to host memory leave alone,
    the padding between sections."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lat = _lattice(*shape, precision)
    ud = inputs.edge_array(*shape, 1.0, 1.0, 1.0, 1.0)
    lat.substeps(12, 1, ud, ud)
    nb = lat.state_bytes()
    fills = (7, 200)
    host = [lat.save(np.full(nb, v, np.uint8)) for v in fills]
    dev = []
    for v in fills:
        room = torch.full((nb + 64,), v, dtype=torch.uint8, device="cuda")
        lat.save(room[offset:offset + nb])
        lat.synchronize()
        got = room.cpu().numpy()
        assert (got[:offset] == v).all() and (got[offset + nb:] == v).all()
        dev.append(got[offset:offset + nb])
    kept = [(a == fills[0]) & (b == fills[1]) for a, b in (host, dev)]
    assert np.array_equal(*kept) and 0 < kept[0].sum() < 20 * 256
    assert all(np.array_equal(a, b) for a, b in zip(host, dev))
