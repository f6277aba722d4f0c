"""Results into memory of every kind: fresh pageable pages, page-locked ones, and
device memory, which the call refuses with a status or fills, but never ends in a
signal."""
import ctypes as C

import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def pointer(address):
    return C.cast(C.c_void_p(address), C.POINTER(C.c_double))


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
def test_results_into_device_memory(precision):
    import torch
    n = 5000
    t = W.target(n=(12, 14, 10))
    s = hpic.Sim(t, None, W.run(), precision=precision)
    rng = np.random.default_rng(3)
    p = {k: rng.uniform(0.1, 0.9, n) * t[m] * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: rng.normal(size=n) for k in ("ux", "uy", "uz")})
    p["tau"] = rng.exponential(1.0, n)
    p["id"] = np.arange(n, dtype=np.uint32)
    s.set_particles(p)
    s.step(2)
    for which in ("T", "Bx"):
        want = s.grid(which)
        room = torch.zeros(want.size, dtype=torch.float64, device="cuda")
        rc = hpic.lib().hpic_read_grid(s.h, hpic.GRID[which], pointer(room.data_ptr()))
        torch.cuda.synchronize()
        assert rc == hpic.HPIC_ECUDA or (rc == 0 and np.array_equal(room.cpu().numpy(), want))
        assert np.array_equal(s.grid(which), want)  # and the next call is as before
    want = s.particles()
    m = len(want["id"])
    room = torch.zeros(m, dtype=torch.float64, device="cuda")
    none, got = C.POINTER(C.c_double)(), C.c_int64()
    rc = hpic.lib().hpic_read_particles(s.h, pointer(room.data_ptr()), *[none] * 6,
                                        C.POINTER(C.c_uint32)(), m, C.byref(got))
    torch.cuda.synchronize()
    assert rc == hpic.HPIC_ECUDA or (rc == 0 and np.array_equal(room.cpu().numpy(), want["x"]))
    assert np.array_equal(s.particles()["x"], want["x"])
    s.close()


@pytest.mark.parametrize("size", [1, 8192, 8193, 300_000])
def test_results_keep_to_their_bytes(size):
    """Fresh memory that ends anywhere in a page: what lies before and behind the
    result stays as it is."""
    t = W.target(n=(12, 14, 10))
    s = hpic.Sim(t, None, W.run(), precision=hpic.HPIC_FP64)
    want = s.grid("jx")
    room = np.empty(size + want.size + 3)
    room[:size], room[size + want.size:] = 7.0, 8.0
    rc = hpic.lib().hpic_read_grid(s.h, hpic.GRID["jx"], pointer(room.ctypes.data + 8 * size))
    assert rc == 0 and np.array_equal(room[size:size + want.size], want)
    assert np.all(room[:size] == 7.0) and np.all(room[size + want.size:] == 8.0)
    s.close()
