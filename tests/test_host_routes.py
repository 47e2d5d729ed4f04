"""Which memory the library's host code hands to kernels and which it copies:
memory of another device is copied, not dereferenced.  On a recording stand-in
for the CUDA runtime (no GPU, kernels not run)."""
import ctypes

import pytest

import fake_cuda
from fake_cuda import DEVICE, HOST, MANAGED


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_cuda.load(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("kind,device,copied", [(DEVICE, 0, False), (MANAGED, 0, False),
                                                (DEVICE, 1, True), (HOST, 0, True)])
@pytest.mark.parametrize("nex,ney", [(20, 10), (700, 330)])  # by tiles, over all nodes
def test_dirichlet_values_of_a_continuum_step(fake, nex, ney, kind, device, copied):
    from paper_1601_02708_gb300._lib import FemParams
    p = FemParams(nex=nex, ney=ney, hx=0.1, hy=0.1, D=1.0, theta=0.5, dt=0.1)
    nodes = (ctypes.c_int * 5)(*range(5))
    h = ctypes.c_void_p()
    assert fake.lib.lbm_fem_init(ctypes.byref(h), ctypes.byref(p), None, 5, nodes, None, None) == 0
    vals = fake.buffer(5 * 8, kind, device)
    fake.clear()
    fake.lib.lbm_fem_step(h, vals)  # (no kernel runs: it reports no convergence)
    assert fake.launched("k_bicgstab_tile" if nex < 100 else "k_bicgstab")
    assert any(s == ctypes.addressof(vals) and n == 40 for _, s, n in fake.copies()) == copied
    fake.lib.lbm_fem_destroy(h)


@pytest.mark.parametrize("kind,device,copied", [(DEVICE, 0, False), (MANAGED, 0, False),
                                                (DEVICE, 1, True), (HOST, 0, True)])
@pytest.mark.parametrize("what", ["lbm_get_populations", "lbm_adjoint"])
def test_fields_read_out(fake, what, kind, device, copied):
    """(outlet_breakthrough reads dJ/dk into memory where its rate field is)"""
    h = fake.lattice(40, 30)
    out = fake.buffer(9 * 40 * 30 * 8, kind, device)
    fake.clear()
    if what == "lbm_adjoint":
        bytes_ = 40 * 30 * 8
        st = fake.lib.lbm_adjoint(h, 2, 1, 0, None, None, None, None, out, None, None, None, None)
    else:
        bytes_ = 9 * 40 * 30 * 8
        st = fake.lib.lbm_get_populations(h, out)
    assert st == 0
    assert any(d == ctypes.addressof(out) and n == bytes_ for d, _, n in fake.copies()) == copied
    fake.lib.lbm_destroy(h)


@pytest.mark.parametrize("kind,device,waits", [(DEVICE, 0, 0), (MANAGED, 0, 0), (DEVICE, 1, 1)])
def test_save_into_device_memory(fake, kind, device, waits):
    """It queues copies and returns, so that it can be captured; the header does
    not travel from the call's stack unless the call waits (another device)."""
    h = fake.lattice(40, 30)
    n = fake.state_bytes(h)
    blob = fake.buffer(n, kind, device)
    fake.clear()
    fake.lib.lbm_save.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t]
    assert fake.lib.lbm_save(h, blob, n) == 0
    assert fake.waits() == waits
    header = any(d == ctypes.addressof(blob) for d, _, _ in fake.copies())
    assert header == (waits > 0) and fake.launched("k_copy_list") == (waits == 0)
    fake.lib.lbm_destroy(h)


@pytest.mark.parametrize("passes", [0, 5])
def test_state_restored_into_a_fresh_slab(fake, passes):
    """The first pass over every node starts with its block counter at zero, and
    is not run on a state that has passes behind it."""
    import numpy as np
    from paper_1601_02708_gb300._lib import Params
    p = Params(nx=40, ny=30, precision=64, tau=0.8, react_mode=1, k_scalar=0.1, dissolution=1)
    h = ctypes.c_void_p()
    assert fake.lib.lbm_init_slab(ctypes.byref(h), ctypes.byref(p), 0, 12, None, None, None, None, None, None) == 0
    n = fake.state_bytes(h)
    fake.lib.lbm_save.argtypes = fake.lib.lbm_restore.argtypes = [ctypes.c_void_p, ctypes.c_void_p,
                                                                  ctypes.c_size_t]
    blob = np.zeros(n, np.uint8)
    assert fake.lib.lbm_save(h, blob.ctypes.data, n) == 0
    up = lambda b: -(-b // 256) * 256
    plane = 160 * 14
    # from the end: flip steps, minerals and nodes of the surface list, the words
    at = n - up(4 * plane) - up(8 * 480) - up(4 * 480) - 256
    blob[at:at + 16].view(np.int32)[:] = (0, 7, 7, passes)
    assert fake.lib.lbm_restore(h, blob.ctypes.data, n) == 0
    fake.clear()
    assert fake.lib.lbm_step_dissolve(h) == 0
    assert fake.launched("lbm_dissolve_dense") == (passes == 0) and not fake.launched("lbm_dissolve_list")
    back = np.zeros(n, np.uint8)
    assert fake.lib.lbm_save(h, back.ctypes.data, n) == 0
    assert list(back[at:at + 16].view(np.int32)) == [0, 0 if passes == 0 else 7, 7, passes]
    fake.clear()
    assert fake.lib.lbm_step_stream(h, 1, 1, 1) == 0 and fake.lib.lbm_step_dissolve(h) == 0
    assert fake.launched("lbm_dissolve_list")
    fake.lib.lbm_destroy(h)
