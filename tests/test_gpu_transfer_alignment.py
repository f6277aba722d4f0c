"""Page-locked arrays cut from one block at any byte: those that do not start at a
multiple of their element's size are copied, the others cross by the kernels."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "z", "ux", "uy", "uz", "tau")


def cut(n, offset):
    """Eight arrays one behind the other in a page-locked block: the ids, then the
    doubles, all of them `offset` bytes past a multiple of their size."""
    import torch
    block = torch.empty(64 + 4 * n + 8 + 7 * 8 * n + 64, dtype=torch.uint8, pin_memory=True).numpy()
    out, at = {}, offset % 4
    out["id"] = np.frombuffer(block.data, np.uint32, n, at)
    at = (at + 4 * n + 7) // 8 * 8 + offset
    for k in KEYS:
        out[k] = np.frombuffer(block.data, np.float64, n, at)
        at += 8 * n
    return out


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
@pytest.mark.parametrize("offset", [0, 4, 1, 6])
def test_arrays_at_any_byte(precision, offset):
    n = 5001
    t = W.target(n=(9, 12, 10))
    rng = np.random.default_rng(offset)
    f = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    p = {k: f(rng.uniform(0, t[m], n)) * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: f(rng.normal(0, 3, n)) for k in ("ux", "uy", "uz")})
    p["tau"] = f(rng.exponential(1.0, n))
    p["id"] = np.arange(n, dtype=np.uint32)
    s = hpic.Sim(t, None, W.run(), precision=precision)
    given, room = cut(n, offset), cut(n, offset)
    for k, v in p.items():
        given[k][:] = v
        room[k][:] = 0
    s.set_particles(given)
    for got in (s.particles(), s.particles(room)):
        assert np.array_equal(got["id"], p["id"])
        for k in KEYS:  # cells and back: two roundings in double of an FP32 value
            assert np.max(np.abs(got[k] - p[k])) <= 4e-16 * np.max(np.abs(p[k])), k
    s.close()


def test_array_across_two_registrations():
    """Arrays whose two ends are page-locked and whose middle is not: the ends alone do
    not make them page-locked.  They are copied, or the copy is refused with a status."""
    import torch
    rt = torch.cuda.cudart()
    torch.cuda.init()
    page = 1 << 16
    n = 3 * page // 8
    t = W.target(n=(9, 12, 10))
    raw = np.empty(8 * 4 * page, np.uint8)
    base = -raw.ctypes.data % page
    rng = np.random.default_rng(2)
    p = {k: rng.uniform(0.1, 0.9, n) * t[m] * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: rng.normal(size=n) for k in ("ux", "uy", "uz")})
    p["tau"] = rng.exponential(1.0, n)
    p["id"] = np.arange(n, dtype=np.uint32)
    given = dict(p, x=np.frombuffer(raw.data, np.float64, n, base))
    given["x"][:] = p["x"]
    first = raw.ctypes.data + base
    for at in (first, first + 2 * page):
        assert int(rt.cudaHostRegister(at, page, 0)) == 0
    try:
        s = hpic.Sim(t, None, W.run(), precision=hpic.HPIC_FP64)
        s.set_particles(p)
        want = s.particles()
        try:
            s.set_particles(given)
        except hpic.HpicError as e:
            assert e.code == hpic.HPIC_ECUDA
        got = s.particles()
        assert all(np.array_equal(got[k], want[k]) for k in KEYS + ("id",))
        s.close()
    finally:
        for at in (first, first + 2 * page):
            rt.cudaHostUnregister(at)
