"""Read-back into destinations of every kind: fresh pages, pages written
before, an address inside a page, a buffer larger than the field. The same
values arrive and nothing beside them changes."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_05448_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


@pytest.mark.parametrize("n", [16, 72])  # below and above the size whose pages are populated ahead
def test_destinations(lbm, n):
    g = lbm.Lattice(n, n, n, 0.6, storage="f32")
    g.init_velocity(workloads.noise_velocity((n, n, n), 0.02, seed=3))
    g.step(2)
    ref = g.macro()[1].reshape(-1)
    need = ref.nbytes
    for touched in (False, True):
        for shift in (0, 8, 4088):  # bytes into the buffer
            for extra in (0, 12345):  # bytes told to the call beyond the field
                raw = np.empty(need + shift + extra + 64, dtype=np.uint8)
                head, tail = slice(0, shift), slice(shift + need, None)
                if touched:
                    raw[:] = 0xa5
                raw[head] = 0x5a
                raw[tail] = 0x5a
                rc = g.L.lbm_get_field(g.h, lbm.FIELD_U, ctypes.c_void_p(raw.ctypes.data + shift), need + extra)
                assert rc == lbm.LBM_OK
                assert np.array_equal(raw[shift:shift + need].copy().view(np.float64), ref)
                assert np.all(raw[head] == 0x5a) and np.all(raw[tail] == 0x5a)
    assert g.L.lbm_get_field(g.h, lbm.FIELD_U, ctypes.c_void_p(raw.ctypes.data), need - 1) == lbm.LBM_EINVAL
    g.close()
