"""The unbounded medium has nothing in it whose sums depend on an order, so its
electrons are the same to the bit whether a run sorts (its steps then are plain, key
the next sort or sort) or not, and as a target of a batch."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

from parity import PKEYS, by_id

pytestmark = pytest.mark.gpu

PHYSICS = hpic.HPIC_DRAG | hpic.HPIC_SCATTER | hpic.HPIC_BREM | hpic.HPIC_UNBOUNDED


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
@pytest.mark.parametrize("n,material", [(33, ["C", "H"]), (30_011, ["Au"]), (30_011, ["C", "H"])])
def test_same_electrons_in_every_kind_of_step(precision, n, material):
    t = W.compound([(m, None) for m in material], n=(12, 10, 14))
    run = W.run(seed=5, physics=PHYSICS, max_history=8)
    rng = np.random.default_rng(n)
    p = {k: rng.uniform(-1, 1 + t[m], n) * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: rng.normal(size=n) * 5 for k in ("ux", "uy", "uz")})
    p["ux"][: n // 10] *= 0.02  # slow ones, some below the tracking cut before long
    p["uy"][: n // 10] *= 0.02
    p["uz"][: n // 10] *= 0.02
    p["tau"] = rng.exponential(0.02, n)
    p["id"] = np.arange(n, dtype=np.uint32)
    out = []
    for interval in (0, 1, 2, 5):
        s = hpic.Sim(t, None, run, precision=precision, sort_interval=interval)
        s.set_particles(p)
        s.step(7)
        out.append((s.particles(), s.tallies()))
        s.close()
    for interval in (0, 3):
        b = hpic.Batch([t], None, run, precision=precision, spare_slots=n, sort_interval=interval)
        b.target(0).set_particles(p)
        b.step(7)
        out.append((b.target(0).particles(), b.target(0).tallies()))
        b.close()
    want, tallies = by_id(out[0][0]), out[0][1]
    # no field, no work: what W_field holds is the difference of two roundings of one
    # energy, at most two last places of it in each of the steps
    u = 2.0**-24 if precision == hpic.HPIC_FP32_MIXED else 2.0**-53
    energy = sum(tallies[k] for k in ("E_live", "E_drag", "E_xray"))
    for _, tb in out:
        assert abs(tb.pop("W_field")) <= 7 * 4 * u * energy
    assert n // 2 < len(want["id"]) <= n and np.unique(want["id"]).size == len(want["id"])
    for other, tb in out[1:]:
        got = by_id(other)
        for k in PKEYS + ("id",):
            assert np.array_equal(got[k], want[k]), k
        for k in tb:  # sums of the same values in another order
            assert np.allclose(tallies[k], tb[k], rtol=1e-6 if precision == hpic.HPIC_FP32_MIXED else 1e-12, atol=0), k
