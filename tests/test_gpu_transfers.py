"""Electrons in and out through page-locked and pageable host arrays (and a mix
of both), at the edges of the transfer kernels' chunks, with dead slots."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "z", "ux", "uy", "uz", "tau")


def pinned(p):
    import torch
    out = {k: torch.empty(len(v), dtype=torch.float64, pin_memory=True).numpy() for k, v in p.items() if k != "id"}
    out["id"] = torch.empty(len(p["id"]), dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)
    for k, v in p.items():
        out[k][:] = v
    return out


def electrons(n, t, seed=1):
    rng = np.random.default_rng(seed)
    f = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    p = {k: f(rng.uniform(0, t[m], n)) * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: f(rng.normal(0, 3, n)) for k in ("ux", "uy", "uz")})
    p["tau"] = f(rng.exponential(1.0, n))
    p["id"] = np.arange(n, dtype=np.uint32)
    p["x"][:1] = 0.0
    p["y"][-1:] = t["ny"] * t["dx"]  # the walls themselves are inside
    return p


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 2047, 2048, 2049, 70001])
def test_round_trip(precision, n):
    t = W.target(n=(9, 12, 10))
    s = hpic.Sim(t, None, W.run(), precision=precision)
    p = electrons(n, t)
    room = pinned({k: np.zeros(n) if k != "id" else np.zeros(n, np.uint32) for k in KEYS + ("id",)})
    mixed = pinned(p)
    mixed.update({k: p[k] for k in ("y", "tau", "id")})
    for given in (p, pinned(p), mixed):
        s.set_particles(given)
        for got in (s.particles(), s.particles(room)):
            assert np.array_equal(got["id"], p["id"])
            for k in KEYS:  # cells and back: two roundings in double of an FP32 value
                assert np.max(np.abs(got[k] - p[k])) <= 4e-16 * np.max(np.abs(p[k])), k
    s.close()


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
def test_lost_electrons_are_left_out(precision):
    """Electrons of an energy below the cut die in the first step: a third of them, in a pattern."""
    t = W.target(n=(9, 12, 10))
    s = hpic.Sim(t, None, W.run(), precision=precision)
    p = electrons(5000, t)
    dead = np.arange(5000) % 3 == 1
    for k in ("ux", "uy", "uz"):
        p[k][dead] = 1e-3
    s.set_particles(pinned(p))
    s.step(1)
    room = pinned({k: np.zeros(5000) if k != "id" else np.zeros(5000, np.uint32) for k in KEYS + ("id",)})
    a, b = s.particles(), s.particles(room)
    assert len(a["id"]) == s.n and set(a["id"]) <= set(p["id"][~dead])
    for k in KEYS + ("id",):
        assert np.array_equal(a[k], b[k]), k
    s.close()


@pytest.mark.parametrize("where", ["pageable", "pinned"])
def test_refused_arrays_leave_the_population(where):
    t = W.target(n=(9, 12, 10))
    s = hpic.Sim(t, None, W.run(), precision=hpic.HPIC_FP32_MIXED)
    p = electrons(3000, t)
    s.set_particles(p)
    before = s.particles()
    L = t["nx"] * t["dx"]
    for k, v in (("x", -1e-12), ("x", L * (1 + 1e-9)), ("z", np.nan), ("y", np.inf), ("id", 0xFFFFFFFF)):
        q = {a: b.copy() for a, b in p.items()}
        q[k][1234] = v
        with pytest.raises(hpic.HpicError):
            s.set_particles(pinned(q) if where == "pinned" else q)
        after = s.particles()
        assert all(np.array_equal(after[a], before[a]) for a in KEYS + ("id",))
    s.close()
