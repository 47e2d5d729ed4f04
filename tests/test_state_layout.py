"""Saved states do not depend on the device's number of SMs, states of the
earlier form are read, and a state whose header claims more partial sums than it
holds is refused.  On a recording stand-in for the CUDA runtime (no GPU)."""
import ctypes

import numpy as np
import pytest

import fake_cuda

SIZES = [(256, 64), (200, 33), (64, 17), (700, 512)]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    f = fake_cuda.load(str(tmp_path_factory.mktemp("fake")))
    for fn in (f.lib.lbm_save, f.lib.lbm_restore):
        fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t]
    return f


def _save(fake, h):
    blob = np.zeros(fake.state_bytes(h), np.uint8)
    assert fake.lib.lbm_save(h, blob.ctypes.data, blob.size) == 0
    return blob


def _partials(nx, ny, rows):
    """Bytes before the partial sums of an FP64 state, their number for
    blocks of 32 x rows, and the size of their section."""
    up = lambda b: -(-b // 256) * 256
    plane = max((nx + 47) // 32 * 32, 160) * max(ny + 2, 10)
    before = 256 + up(72 * plane) + up(4 * plane) + up(8 * plane) + up(16 * (nx + ny)) + up(8 * ny)
    n = max(-(-nx // 32) * -(-ny // rows), -(-nx // 96) * -(-ny // 8)) + 1
    return before, n, up(8 * n)


@pytest.mark.parametrize("nx,ny", SIZES)
def test_size_on_any_device(fake, nx, ny):
    """(FP64; the FP32 lattice runs the same blocks on every device)"""
    sizes = set()
    for sms in (152, 148, 40, 2):
        fake.lib.fake_sms(sms)
        h = fake.lattice(nx, ny)
        sizes.add(fake.state_bytes(h))
        fake.lib.lbm_destroy(h)
    fake.lib.fake_sms(152)
    assert len(sizes) == 1


@pytest.mark.parametrize("sms", [152, 2])
@pytest.mark.parametrize("old_rows", [2, 8])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_states_of_the_earlier_form(fake, nx, ny, old_rows, sms):
    fake.lib.fake_sms(sms)
    h = fake.lattice(nx, ny)
    state = np.random.default_rng(nx).integers(0, 256, fake.state_bytes(h)).astype(np.uint8)
    state[:256] = _save(fake, h)[:256]
    before, n, section = _partials(nx, ny, 2)
    head = state[:48].view(np.int32)  # magic 0-1, steps 2-3, nx, ny, precision, dissolution, nparts
    _, old_n, old_section = _partials(nx, ny, old_rows)
    head[8] = old_n - 1
    old = np.concatenate([state[:before], state[before:before + old_section], state[before + section:]])
    old[0] = ord("5")
    assert fake.lib.lbm_restore(h, old.ctypes.data, old.size) == 0, fake.lib.lbm_last_error()
    back = _save(fake, h)
    inner = slice(before, before + 8 * old_n)
    assert np.array_equal(back[inner], old[inner])
    # the sections behind the partial sums: the outlet's fluxes, the counters
    got, want = back[before + section:], state[before + section:]
    counters = slice(-(-8 * ny // 256) * 256, -(-8 * ny // 256) * 256 + 32)
    assert np.array_equal(got[:8 * ny], want[:8 * ny]) and np.array_equal(got[counters], want[counters])
    plane = slice(256, 256 + 72 * (before // 100 // 72))
    assert np.array_equal(back[plane], old[plane])
    assert back[:48].view(np.int32)[8] == old_n - 1
    fake.lib.lbm_destroy(h)
    fake.lib.fake_sms(152)


@pytest.mark.parametrize("nparts", [-1, 1 << 20])
def test_more_partial_sums_than_held(fake, nparts):
    h = fake.lattice(256, 64)
    blob = _save(fake, h)
    blob[:48].view(np.int32)[8] = nparts
    assert fake.lib.lbm_restore(h, blob.ctypes.data, blob.size) == -5  # LBM_ERR_STATE
    fake.lib.lbm_destroy(h)
